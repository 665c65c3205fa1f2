// cgkern.cuh -- device building blocks shared by the CG kernels (graph-launched and
// persistent): deterministic reductions, the product rows of one slice, shape dispatch.
#pragma once

#include <type_traits>

#include "common.cuh"
#include "ptx.cuh"

namespace gb {

constexpr int kCgBlock = 256;    // CTAs of the kernels around the iteration (residual, start)
constexpr int kCgCtasPerSm = 4;  // at most this many of them per SM

int cg_grid(int32_t n);

// The kernels of an iteration run one CTA per SM, as many threads as the work needs (64 to
// kIterThreads): that leaves 152 partial sums, few enough for every CTA of the next kernel to
// add them itself, and small systems still spread over every SM's FP64 pipe (2 operations per
// SM and clock).
//
// A lane of the product holding at most 16 bytes of values per entry keeps pq_unroll = 5
// entries in flight (a whole row of the tetrahedral meshes) at 1,024 threads per SM and 64
// registers -- measured on the 6M-row mesh against two entries at 1,536 threads (40
// registers): FP64 CG 185 -> 176 us per iteration, the FP32 refinement solve 4.7 % faster;
// wider lanes keep two entries, and so do matrices whose widest slice has no fewer load_rounds in
// fives than in twos.  (That count charges a round's missing entries, which are masked here but
// still take the FP64 pipe: us per FP64 iteration of 3M rows, two / five in flight, rows of 3
// entries 82 / 88, 4 85 / 90, 8 107 / 113, 9 117 / 115, 5 95 / 88.)
constexpr int kIterThreads = 1024;
constexpr int pq_min_ctas(int value_bytes) { return value_bytes >= 64 ? 3 : 4; }
constexpr int pq_unroll(int value_bytes) { return value_bytes <= 16 ? 5 : 2; }
bool cg_pq_deep(const spmv_matrix_t A, int uu);

// Grid of an iteration kernel over `items` slice-lanes or 16-byte vectors: CTA c takes the `chunk`
// items from c * chunk, its thread t those t, t + threads, ... into the chunk.  Equal contiguous
// chunks, since a grid stride leaves the last, partly filled round of items to some of the SMs:
// the 6M-row product takes 19.3 rounds of 152 x 1,024 items, 20 on a third of the SMs.  The grid
// fixes the order of the reductions, so it depends on the handle and the device only; the
// persistent kernel uses the same grid and gives identical results.
struct IterGrid {
    int ctas, threads;
    int64_t chunk;
    bool operator==(const IterGrid &o) const {
        return ctas == o.ctas && threads == o.threads && chunk == o.chunk;
    }
    bool single() const { return chunk <= threads; }  // a thread for every item
};
// first item and end of the calling thread's items
__device__ __forceinline__ int64_t iter_begin(int64_t chunk) {
    return (int64_t)blockIdx.x * chunk + threadIdx.x;
}
__device__ __forceinline__ int64_t iter_end(int64_t chunk, int64_t items) {
    const int64_t e = ((int64_t)blockIdx.x + 1) * chunk;
    return e < items ? e : items;
}
// The calling thread's place in an IterGrid each of whose CTAs is run by Q smaller ones (a
// solve beside others, see IterForm); Q = 1: the grid as it is.
template <int Q>
struct IterSlot {
    int cta, id;   // CTA of the grid, thread of it
    bool in;       // whether the grid has that thread
    __device__ __forceinline__ explicit IterSlot(int threads) {
        cta = (int)blockIdx.x / Q;
        id = (int)(blockIdx.x % Q * blockDim.x + threadIdx.x);
        in = Q == 1 || id < threads;
    }
    __device__ __forceinline__ int64_t begin(int64_t chunk) const { return cta * chunk + id; }
    __device__ __forceinline__ int64_t end(int64_t chunk, int64_t items) const {
        const int64_t e = (cta + 1) * chunk;
        return !in ? 0 : e < items ? e : items;
    }
};
// What an iteration leaves in L2 for the next one.  The matrix is streamed evict-first unless it
// and the vectors fit (three quarters of) the L2 together; the vectors that a FP32 sweep is the
// last to touch are, unless the five vectors take no more than half of it.  Per FP32 iteration,
// evict-first / kept: matrix 1.5M rows 23.1 / 21.3 us (75 MB in all; 2.1M rows, 103 MB: 27.8 /
// 30.8), vectors 2.1M rows 29.1 / 27.8, 3.1M (61 MB) 35.6 / 34.5 (4.4M: 50.2 / 51.5).
struct IterKeep {
    bool matrix, vectors;
};
IterKeep cg_keep(const spmv_matrix_t A, int elem_bytes, int solves = 1);  // that share the L2

IterGrid cg_iter_grid(int64_t items, int max_threads);
IterGrid cg_pq_grid(const spmv_matrix_t A, int L, int value_bytes);
IterGrid cg_sweep_grid(const spmv_matrix_t A, int vec);

// Hint: bring the line holding p into L1 without waiting for it (a later load of it hits).
__device__ __forceinline__ void prefetch_l1(const void *p) {
    asm volatile("prefetch.global.L1 [%0];" ::"l"(p));
}

// Sum over the CTA in a fixed tree; the total is left in every lane of warp 0.
template <int NV>
__device__ __forceinline__ void block_sum(double (&v)[NV]) {
    __shared__ double sh[NV][kCgBlock / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v[k] += __shfl_xor_sync(0xffffffffu, v[k], o);
    }
    __syncthreads();
    if (lane == 0) {
#pragma unroll
        for (int k = 0; k < NV; ++k) sh[k][warp] = v[k];
    }
    __syncthreads();
    if (warp == 0) {
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            double t = lane < kCgBlock / 32 ? sh[k][lane] : 0.0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
            v[k] = t;
        }
    }
}

// ---- reductions of the iteration kernels ----------------------------------------------------
// Sums over threads and CTAs are formed in fixed point: the values of a warp are aligned to
// the largest exponent among them, cut into three 22-bit limbs and added by the integer warp
// reductions (redux.sync).  The sum is exact but for the bits of a value that lie more than 64
// below the largest value's leading one, so it is no further from the true sum than a tree of
// FP64 additions, it does not depend on the order, and it leaves the SM's FP64 pipe alone: summing
// a CTA takes 710 clocks with 64 threads and 1,200 with 1,024 where FP64 shuffle trees take 1,530
// and 4,510 (a warp-wide FP64 addition holds the pipe for 16 clocks).  FP64 iteration of a
// 304K-row system 15.5 -> 14.7 us, FP32 11.5 -> 10.8 us, 1M rows FP32 18.7 -> 17.6 us; over random
// summands of mixed signs and magnitudes the error against long double, relative to the sum of
// magnitudes, is 1.0e-16 at worst where an FP64 tree has 2.6e-16.
constexpr int kFxLimb = 22;
constexpr int kFxMask = (1 << kFxLimb) - 1;
constexpr int kFxBad = 0x7ff;  // exponent field of infinities and NaN

// (l2 2^44 + l1 2^22 + l0) 2^(e - 1086), e a biased FP64 exponent; e = kFxBad: not finite
struct Fx {
    int l0, l1, l2, e;
};

// biased FP64 exponent (at least 1) and the significand with its leading one in bit 63
__device__ __forceinline__ void fx_split(double a, int &e, uint64_t &m) {
    const uint64_t b = (uint64_t)__double_as_longlong(a);
    const int f = (int)((b >> 52) & 0x7ff);
    m = (b << 12) >> 1 | (f ? 1ull << 63 : 0ull);
    e = f ? f : 1;
}
__device__ __forceinline__ void fx_split(float a, int &e, uint64_t &m) {
    const uint32_t b = __float_as_uint(a);
    const int f = (int)((b >> 23) & 0xff);
    m = (uint64_t)((b << 9) >> 1 | (f ? 1u << 31 : 0u)) << 32;
    e = f == 0xff ? kFxBad : (f ? f : 1) + 896;
}

// -1 for a negative value, else 0
__device__ __forceinline__ int fx_sign(double a) { return __double2hiint(a) >> 31; }
__device__ __forceinline__ int fx_sign(float a) { return __float_as_int(a) >> 31; }

// The sum of the calling warp's values (M per lane), in every lane.  M <= 8.
template <int M, typename T>
__device__ __forceinline__ Fx fx_warp(const T (&a)[M]) {
    int e[M];
    uint64_t m[M];
    int top = 0;
#pragma unroll
    for (int j = 0; j < M; ++j) {
        fx_split(a[j], e[j], m[j]);
        top = e[j] > top ? e[j] : top;
    }
    Fx s;
    s.e = __reduce_max_sync(0xffffffffu, top);
    s.l0 = s.l1 = s.l2 = 0;
#pragma unroll
    for (int j = 0; j < M; ++j) {
        const int sh = s.e - e[j];
        const uint64_t v = sh < 64 ? m[j] >> sh : 0ull;
        const int neg = fx_sign(a[j]);
        s.l0 += (((int)v & kFxMask) ^ neg) - neg;
        s.l1 += (((int)(v >> kFxLimb) & kFxMask) ^ neg) - neg;
        s.l2 += ((int)(v >> (2 * kFxLimb)) ^ neg) - neg;
    }
    s.l0 = __reduce_add_sync(0xffffffffu, s.l0);
    s.l1 = __reduce_add_sync(0xffffffffu, s.l1);
    s.l2 = __reduce_add_sync(0xffffffffu, s.l2);
    return s;
}

// The sum of the lanes' fx_warp sums (of one value per lane), in every lane.
__device__ __forceinline__ Fx fx_combine(const Fx &f) {
    Fx s;
    s.e = __reduce_max_sync(0xffffffffu, f.e);
    const int sh = s.e - f.e;
    // the value as rest 2^32 + low, shifted down to the common exponent
    const int64_t h = ((int64_t)f.l2 << kFxLimb) + f.l1 + (f.l0 >> kFxLimb);
    const uint32_t low = (uint32_t)(f.l0 & kFxMask) | ((uint32_t)h << kFxLimb);
    const int64_t rest = h >> (32 - kFxLimb);
    const uint32_t w = sh < 32 ? __funnelshift_r(low, (uint32_t)rest, sh)
                               : (uint32_t)(rest >> (sh - 32 < 63 ? sh - 32 : 63));
    const int64_t r = rest >> (sh < 63 ? sh : 63);
    s.l0 = (int)w & kFxMask;
    s.l1 = (int)(w >> kFxLimb | (uint32_t)r << (32 - kFxLimb)) & kFxMask;
    s.l2 = (int)(r >> (2 * kFxLimb - 32));
    s.l0 = __reduce_add_sync(0xffffffffu, s.l0);
    s.l1 = __reduce_add_sync(0xffffffffu, s.l1);
    s.l2 = __reduce_add_sync(0xffffffffu, s.l2);
    return s;
}

// The value rounded to FP64 (NaN when a summand was not finite).
__device__ __forceinline__ double fx_value(const Fx &f) {
    if (f.e == kFxBad) return __longlong_as_double(0x7ff8000000000000ll);
    // sign and magnitude h 2^22 + low
    int64_t h = ((int64_t)f.l2 << kFxLimb) + f.l1 + (f.l0 >> kFxLimb);
    uint32_t low = (uint32_t)(f.l0 & kFxMask);
    const bool neg = h < 0;
    if (neg) {
        h = -h - (low != 0);
        low = (0u - low) & kFxMask;
    }
    // the leading 64 bits with the leading one in bit 63; its position in the magnitude
    uint64_t x;
    int pos;
    if (h) {
        const int k = 63 - __clzll(h);
        pos = k + kFxLimb;
        x = (uint64_t)h << (63 - k) |
            (k <= 41 ? (uint64_t)low << (41 - k) : (uint64_t)low >> (k - 41));
    } else {
        if (!low) return 0.0;
        pos = 31 - __clz(low);
        x = (uint64_t)low << (63 - pos);
    }
    const int be = pos + f.e - 63;  // biased exponent
    if (be < 1 || be > 2046) {
        const double v = scalbn(fma((double)h, 4194304.0, (double)low), f.e - 1086);
        return neg ? -v : v;
    }
    uint64_t m = x >> 11;
    const uint32_t cut = (uint32_t)x & 0x7ffu;
    m += cut > 0x400u || (cut == 0x400u && (m & 1));
    const uint64_t b = ((uint64_t)(be - 1) << 52) + m;
    return __longlong_as_double((long long)(b | (uint64_t)neg << 63));
}

// Sum of v[k] over the first TT threads of the CTA (TT >= 32 NV, a multiple of 32): quantity
// k's total is returned in every lane of warp k, k < NV.
template <int NV>
struct FoldSmem {
    int4 fx[NV][kIterThreads / 32];
};
template <int NV, int NS, typename T>
__device__ __forceinline__ double fold_block(const T (&v)[NV], int TT, FoldSmem<NS> &sm) {
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    __syncthreads();  // sm may still be read from a previous call
    if (t < TT) {
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            const T one[1] = {v[k]};
            const Fx f = fx_warp<1>(one);
            if (lane == 0) sm.fx[k][warp] = make_int4(f.l0, f.l1, f.l2, f.e);
        }
    }
    __syncthreads();
    double s = 0.0;
    if (warp < NV) {
        Fx f = {0, 0, 0, 0};
        if (32 * lane < TT) {
            const int4 q = sm.fx[warp][lane];
            f = {q.x, q.y, q.z, q.w};
        }
        s = fx_value(fx_combine(f));
    }
    return s;
}

// Sum of one value per CTA (at most 32 kPartLoads CTAs) by one warp: lane l holds the values
// of CTAs l, l + 32, ...
constexpr int kPartLoads = 5;
__device__ __forceinline__ double sum_parts(const double (&a)[kPartLoads]) {
    return fx_value(fx_warp<kPartLoads>(a));
}

// Where the CTAs that share one of an IterGrid leave their warps' sums.
struct SplitSums {
    int4 fx[32 * kPartLoads][2][kIterThreads / 32];
    unsigned arrived[32 * kPartLoads];
};

// The sums of v over a CTA of the grid, to part[k * ctas + cta].  Of Q CTAs that share it the last
// one to arrive adds what all their warps left, in the order and with the bits of a single one.
template <int Q, int NV, typename T>
__device__ __forceinline__ void store_parts(const IterSlot<Q> &slot, int threads, const T (&v)[NV],
                                            SplitSums *split, double *part) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if constexpr (Q == 1) {
        __shared__ FoldSmem<NV> sm;
        const double s = fold_block<NV>(v, blockDim.x, sm);
        if (warp < NV && lane == 0) part[warp * gridDim.x + blockIdx.x] = s;
    } else {
        __shared__ bool last;
#pragma unroll
        for (int k = 0; k < NV; ++k) {
            const T one[1] = {v[k]};
            const Fx f = fx_warp<1>(one);
            if (lane == 0 && slot.in)
                split->fx[slot.cta][k][slot.id >> 5] = make_int4(f.l0, f.l1, f.l2, f.e);
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            last = atomicAdd(&split->arrived[slot.cta], 1u) == Q - 1;
            if (last) split->arrived[slot.cta] = 0u;
            __threadfence();
        }
        __syncthreads();
        if (last && warp < NV) {
            Fx f = {0, 0, 0, 0};
            if (32 * lane < threads) {
                const int4 q = ld_l2(&split->fx[slot.cta][warp][lane]);
                f = {q.x, q.y, q.z, q.w};
            }
            const double s = fx_value(fx_combine(f));
            if (lane == 0) part[warp * (gridDim.x / Q) + slot.cta] = s;
        }
    }
}

// The scalars of an iteration from its sums, computed by one thread of each CTA and shared: an
// FP64 division is some twenty operations, which all 32 warps of a CTA would put through the
// SM's 2-per-clock pipe in 3 us.
template <typename T>
struct StepScalars {
    double rr;
    T coef;    // alpha, or beta
    int done;  // 0, or the reason to stop after this step (CgScalars::done)
};

// alpha = rho / (p.q); done = 3 when it does not exist
template <typename T>
__device__ __forceinline__ void step_alpha(double rho, double pq, StepScalars<T> &s) {
    s.done = (pq == 0.0 || !isfinite(pq)) ? 3 : 0;
    s.coef = (T)(rho / pq);
}
// beta = r.z / rho, from the sums r.z and r.r
template <typename T>
__device__ __forceinline__ void step_beta(double rho, double rz, StepScalars<T> &s) {
    s.coef = (T)(rz / rho);
}
__device__ __forceinline__ int step_done(double rr, double limit, int iters, int max_iter) {
    return rr <= limit ? 1 : (!isfinite(rr) ? 3 : (iters >= max_iter ? 2 : 0));
}

// Sum over i < count of part[i], by the calling warp (in every lane).  The kernels of a CG
// iteration leave their CTAs' sums in part and each CTA of the next kernel adds them up: one
// read of a few KB from L2, where a last-CTA reduction costs a fence, an atomic ticket and a
// second pass at the end of every kernel.
__device__ __forceinline__ double reduce_parts(const double *part, int count) {
    const int lane = threadIdx.x & 31;
    double a[kPartLoads];
#pragma unroll
    for (int j = 0; j < kPartLoads; ++j)
        a[j] = lane + 32 * j < count ? ld_l2(part + lane + 32 * j) : 0.0;
    return sum_parts(a);
}

// Each CTA stores its partial sums in part[k * gridDim.x + cta]; the CTA that arrives last
// (atomic ticket) sums all partials in a fixed order.  Returns true in that CTA, with the
// grid totals in tot[] (valid in thread 0); the ticket is reset for the next launch.
template <int NV>
__device__ bool grid_sum_last(double (&v)[NV], double *part, unsigned *ticket, double (&tot)[NV]) {
    __shared__ bool last;
    block_sum<NV>(v);
    if (threadIdx.x == 0) {
#pragma unroll
        for (int k = 0; k < NV; ++k) part[k * gridDim.x + blockIdx.x] = v[k];
        __threadfence();
        last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
    __syncthreads();
    if (!last) return false;
    __threadfence();
    double s[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) {
        s[k] = 0.0;
        for (int i = threadIdx.x; i < (int)gridDim.x; i += kCgBlock)
            s[k] += ld_l2(part + k * gridDim.x + i);
    }
    block_sum<NV>(s);
    if (threadIdx.x == 0) {
#pragma unroll
        for (int k = 0; k < NV; ++k) tot[k] = s[k];
        *ticket = 0u;
    }
    return true;
}

// A slice-lane: R rows of one slice, held by one thread.
struct SliceLane {
    int64_t at;     // first stored entry of the lane's first row
    int w;          // stored entries per row of the slice
    int32_t cbase;  // column base of 16-bit relative columns
};

template <int R, int L, typename ColT>
__device__ __forceinline__ SliceLane slice_open(int64_t g, const int64_t *sp, const ColT &cols) {
    const int64_t slice = g / L;
    const int lane = (int)(g % L);
    const int64_t base = sp[slice];
    SliceLane s;
    s.w = (int)((sp[slice + 1] - base) / (L * R));
    s.cbase = cols.base(slice);
    s.at = base + lane * R;
    return s;
}

// UU stored entries of each of a lane's R rows, in flight together.  MASKED: entries past the
// slice's width are not loaded (column -1).
template <typename T, int R, int UU>
struct SliceRound {
    T v[UU][R];
    int32_t c[UU][R];

    template <int L, bool MASKED = false, typename ColT>
    __device__ __forceinline__ void load(const SliceLane &s, int t, const ColT &cols,
                                         const T *val, uint64_t pol) {
        constexpr int S = L * R;
#pragma unroll
        for (int u = 0; u < UU; ++u) {
            if (!MASKED || t + u < s.w) {
                ld_stream(val + s.at + (int64_t)(t + u) * S, pol, v[u]);
                cols.template load<R>(s.at + (int64_t)(t + u) * S, 0, pol, s.cbase, c[u]);
            } else {
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    v[u][i] = T(0);
                    c[u][i] = -1;
                }
            }
        }
    }

    template <bool COHERENT>
    __device__ __forceinline__ void multiply(const T *x, T (&acc)[R]) const {
        T xv[UU][R];
#pragma unroll
        for (int u = 0; u < UU; ++u)
#pragma unroll
            for (int i = 0; i < R; ++i)
                xv[u][i] = c[u][i] >= 0 ? (COHERENT ? ld_x_coherent(x + c[u][i]) : ld_x(x + c[u][i]))
                                        : T(0);
#pragma unroll
        for (int u = 0; u < UU; ++u)
#pragma unroll
            for (int i = 0; i < R; ++i)
                if (c[u][i] >= 0) acc[i] = fma_t(v[u][i], xv[u][i], acc[i]);
    }
};

// The R row sums of a slice-lane: its entries in column order, fused multiply-add from +0.0,
// padding skipped (the order of spmv_sell).  rd holds the first round when the slice has at
// least UU entries (the caller loads it, as early as it can); the remainder of a row shorter
// than a round is one more round with the missing entries masked.  COHERENT selects coherent
// gathers of x, for kernels in which other CTAs rewrite x between barriers.
template <typename T, int R, int L, bool COHERENT, int UU, typename ColT>
__device__ __forceinline__ void slice_multiply(const SliceLane &s, SliceRound<T, R, UU> &rd,
                                               const ColT &cols, const T *val, const T *x,
                                               uint64_t pol, T (&acc)[R]) {
#pragma unroll
    for (int i = 0; i < R; ++i) acc[i] = T(0);
    int t = 0;
    if (s.w >= UU) {
        rd.template multiply<COHERENT>(x, acc);
        for (t = UU; t + UU <= s.w; t += UU) {
            rd.template load<L>(s, t, cols, val, pol);
            rd.template multiply<COHERENT>(x, acc);
        }
    }
    if (t < s.w) {
        rd.template load<L, true>(s, t, cols, val, pol);
        rd.template multiply<COHERENT>(x, acc);
    }
}

template <typename T, int R, int L, bool COHERENT = false, int UU = 2, typename ColT>
__device__ __forceinline__ void slice_rows(int64_t slice, int lane, const int64_t *sp,
                                           const ColT &cols, const T *val, const T *x,
                                           uint64_t pol, T (&acc)[R]) {
    const SliceLane s = slice_open<R, L>(slice * L + lane, sp, cols);
#pragma unroll
    for (int i = 0; i < R; ++i) acc[i] = T(0);
    int t = 0;
    for (; t + UU <= s.w; t += UU) {
        SliceRound<T, R, UU> rd;
        rd.template load<L>(s, t, cols, val, pol);
        rd.template multiply<COHERENT>(x, acc);
    }
    if (t < s.w) {
        SliceRound<T, R, UU> rd;
        rd.template load<L, true>(s, t, cols, val, pol);
        rd.template multiply<COHERENT>(x, acc);
    }
}

// ---- vector sweeps of one CG iteration (grid-stride, 16-byte vectors, scalar tail) --------
// Shared by the graph-launched kernels and the persistent kernel, so both produce the same
// per-thread partial sums.  Vectors are plain (coherent) loads: inside the persistent kernel
// they are rewritten between grid barriers.
template <typename T>
struct Vec16;
template <>
struct Vec16<double> {
    using type = double2;
    static constexpr int n = 2;
};
template <>
struct Vec16<float> {
    using type = float4;
    static constexpr int n = 4;
};

template <typename T>
__device__ __forceinline__ void vload(const T *p, T (&v)[Vec16<T>::n]) {
    const typename Vec16<T>::type t = *reinterpret_cast<const typename Vec16<T>::type *>(p);
    if constexpr (Vec16<T>::n == 2) {
        v[0] = t.x;
        v[1] = t.y;
    } else {
        v[0] = t.x;
        v[1] = t.y;
        v[2] = t.z;
        v[3] = t.w;
    }
}

template <typename T>
__device__ __forceinline__ void vstore(T *p, const T (&v)[Vec16<T>::n]) {
    typename Vec16<T>::type t;
    if constexpr (Vec16<T>::n == 2) {
        t.x = v[0];
        t.y = v[1];
    } else {
        t.x = v[0];
        t.y = v[1];
        t.z = v[2];
        t.w = v[3];
    }
    *reinterpret_cast<typename Vec16<T>::type *>(p) = t;
}

// 16-byte loads and stores marked evict-first in L2 (and not kept in L1), for the vectors an
// FP32 sweep is the last to touch in its iteration, so that the ones the next kernel reads
// stay in L2: measured on the 6M-row mesh, the FP32 refinement solve 99 -> 94 ms.  The FP64
// sweeps, co-bound by the FP64 pipe, measured slower with the hints (FP64 CG 194 -> 206 ms)
// and keep plain loads and stores.  vload_h / vstore_h pick the form by element type.
__device__ __forceinline__ void vload_ef(const float *p, float (&v)[4], uint64_t pol) {
    asm volatile("ld.global.L1::no_allocate.L2::cache_hint.v4.f32 {%0,%1,%2,%3}, [%4], %5;"
                 : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3])
                 : "l"(p), "l"(pol));
}
__device__ __forceinline__ void vstore_ef(float *p, const float (&v)[4], uint64_t pol) {
    asm volatile("st.global.L2::cache_hint.v4.f32 [%0], {%1,%2,%3,%4}, %5;" ::"l"(p), "f"(v[0]),
                 "f"(v[1]), "f"(v[2]), "f"(v[3]), "l"(pol)
                 : "memory");
}

template <typename T>
__device__ __forceinline__ void vload_h(const T *p, T (&v)[Vec16<T>::n], uint64_t pol) {
    if constexpr (sizeof(T) == 4) vload_ef(p, v, pol);
    else vload(p, v);
}
template <typename T>
__device__ __forceinline__ void vstore_h(T *p, const T (&v)[Vec16<T>::n], uint64_t pol) {
    if constexpr (sizeof(T) == 4) vstore_ef(p, v, pol);
    else vstore(p, v);
}

// One thread's vector of the x/r update.  D^-1 does not change during a solve, so a kernel may
// load it before the kernel it depends on has finished (load_d); the rest comes after.
template <typename T>
struct XrVec {
    static constexpr int V = Vec16<T>::n;
    T x[V], r[V], p[V], q[V], d[V];
    __device__ __forceinline__ void load_d(const T *dinv, int64_t i) { vload(dinv + i, d); }
    __device__ __forceinline__ void load(const T *xg, const T *rg, const T *pg, const T *qg,
                                         int64_t i, uint64_t pol) {
        vload_h(xg + i, x, pol);
        vload(rg + i, r);
        vload(pg + i, p);
        vload_h(qg + i, q, pol);
    }
    // x += alpha p; r -= alpha q; r.(D^-1 r) into vz, r.r into vr
    __device__ __forceinline__ void update(T alpha, T *xg, T *rg, int64_t i, uint64_t pol, T &vz,
                                           T &vr) {
#pragma unroll
        for (int e = 0; e < V; ++e) {
            x[e] = fma_t(alpha, p[e], x[e]);
            r[e] = fma_t(-alpha, q[e], r[e]);
            vz = fma_t(r[e], d[e] * r[e], vz);
            vr = fma_t(r[e], r[e], vr);
        }
        vstore_h(xg + i, x, pol);
        vstore(rg + i, r);
    }
};

// x += alpha p; r -= alpha q over the vectors k = from, from + stride, ... below end (n may cut the
// last one short); accumulates r.(D^-1 r) into vz and r.r into vr.  x and q are not needed again
// in this iteration (pol, in FP32); r, p and D^-1 are read by the p update.
template <typename T, int UNROLL = 4>
__device__ __forceinline__ void sweep_update_xr(int32_t n, int64_t from, int64_t end,
                                                int64_t stride, uint64_t pol, T alpha, T *x,
                                                T *r, const T *p, const T *q, const T *dinv,
                                                T &vz, T &vr) {
    constexpr int V = Vec16<T>::n;
    const int64_t nv = n / V, full = nv < end ? nv : end;
    int64_t k = from;
#pragma unroll UNROLL
    for (; k < full; k += stride) {
        XrVec<T> v;
        v.load(x, r, p, q, k * V, pol);
        v.load_d(dinv, k * V);
        v.update(alpha, x, r, k * V, pol, vz, vr);
    }
    if (k == nv && k < end) {
        for (int64_t i = k * V; i < n; ++i) {
            const T xi = fma_t(alpha, p[i], x[i]);
            const T ri = fma_t(-alpha, q[i], r[i]);
            x[i] = xi;
            r[i] = ri;
            vz = fma_t(ri, dinv[i] * ri, vz);
            vr = fma_t(ri, ri, vr);
        }
    }
}

// One thread's vector of the p update (D^-1 apart, as in XrVec).
template <typename T>
struct PVec {
    static constexpr int V = Vec16<T>::n;
    T r[V], d[V], p[V];
    __device__ __forceinline__ void load_d(const T *dinv, int64_t i, uint64_t pol) {
        vload_h(dinv + i, d, pol);
    }
    __device__ __forceinline__ void load(const T *rg, const T *pg, int64_t i, uint64_t pol) {
        vload_h(rg + i, r, pol);
        vload(pg + i, p);
    }
    __device__ __forceinline__ void update(T beta, T *pg, int64_t i) {
#pragma unroll
        for (int e = 0; e < V; ++e) p[e] = fma_t(beta, p[e], d[e] * r[e]);
        vstore(pg + i, p);
    }
};

// p = D^-1 r + beta p over the vectors k = from, from + stride, ... below end.  r and D^-1 are next read by
// the next iteration's x/r update (pol, in FP32); the new p stays in L2 for the product's
// gathers.
template <typename T, int UNROLL = 4>
__device__ __forceinline__ void sweep_update_p(int32_t n, int64_t from, int64_t end,
                                               int64_t stride, uint64_t pol, T beta, const T *r,
                                               const T *dinv, T *p) {
    constexpr int V = Vec16<T>::n;
    const int64_t nv = n / V, full = nv < end ? nv : end;
    int64_t k = from;
#pragma unroll UNROLL
    for (; k < full; k += stride) {
        PVec<T> v;
        v.load(r, p, k * V, pol);
        v.load_d(dinv, k * V, pol);
        v.update(beta, p, k * V);
    }
    if (k == nv && k < end) {
        for (int64_t i = k * V; i < n; ++i) p[i] = fma_t(beta, p[i], dinv[i] * r[i]);
    }
}

// (R, L) of the sliced kernels for a slice height and value type.
template <typename T, typename F>
spmv_status_t with_shape(int S, F &&f) {
    using std::integral_constant;
    if constexpr (sizeof(T) == 8) {
        switch (S) {
            case 32: return f(integral_constant<int, 1>{}, integral_constant<int, 32>{});
            case 64: return f(integral_constant<int, 2>{}, integral_constant<int, 32>{});
            case 128: return f(integral_constant<int, 4>{}, integral_constant<int, 32>{});
            case 256: return f(integral_constant<int, 8>{}, integral_constant<int, 32>{});
        }
    } else {
        switch (S) {
            case 32: return f(integral_constant<int, 4>{}, integral_constant<int, 8>{});
            case 64: return f(integral_constant<int, 4>{}, integral_constant<int, 16>{});
            case 128: return f(integral_constant<int, 4>{}, integral_constant<int, 32>{});
            case 256: return f(integral_constant<int, 8>{}, integral_constant<int, 32>{});
        }
    }
    return SPMV_ERR_INVALID_ARG;
}

}  // namespace gb
