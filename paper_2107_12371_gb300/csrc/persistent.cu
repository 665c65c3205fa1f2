// persistent.cu -- a whole Jacobi-PCG loop in one cooperative kernel (FP64 solves, and the FP32
// inner solves of iterative refinement).
//
// One CTA per SM (cooperative launch) runs the iterations on the graph path's grids, with the
// same per-CTA partitions and reduction trees, so the results are the graph path's bit for bit.
// The three phases of an iteration (q = A p with p.q; x/r update with r.z and r.r; p update)
// are separated by exchanges: each CTA posts its sums in a slot of its own, value and
// iteration number in one 16-byte word, and one warp of every CTA reads all slots until they
// carry the iteration's number.  A wait and the sum it waits for are thus one round trip to
// L2, and all CTAs hold bit-identical scalars and take identical branch decisions.
//
// Systems with a thread for every 16-byte vector of rows (up to 311K rows in FP64 and 622K in
// FP32 on 152 SMs) whose matrix fits the SMs' shared memory run in the resident form: the
// matrix stays in shared memory, x, r, p and D^-1 in registers, and only p goes to memory for
// the other threads' gathers.  Up to 512 threads per SM its p update needs no exchange of its
// own (PAIRS): each row's pair (D^-1 r, p) is published with the r.z sums, and the next product
// forms beta p + D^-1 r for every entry it gathers, the same operation on the same operands as
// the row's own update.
//
// Measured per iteration against three atomic-counter barriers per iteration on 256-thread CTAs
// (us, whole solve over its iterations): FP64 10K rows 20.4 -> 9.5, 304K 28.5 -> 18.7, 1M 56.3
// -> 40.1, 6M 188 -> 164; FP32 inner iterations 304K 21.8 -> 12.5, 6M 82.3 -> 70.2.
//
// Every wait is bounded: after 2 s without progress the waiting CTA records done = 4 (timeout)
// and leaves; the others then leave by their own limits, so a fault can never leave the GPU
// spinning.  Vectors that change while the kernel runs are read with coherent loads only (never
// through the read-only .nc path).
#include <algorithm>

#include "cgkern.cuh"

namespace gb {
namespace {

__device__ __forceinline__ long long global_timer_ns() {
    long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

constexpr long long kWaitLimitNs = 2000000000LL;

// A slot: a sum (its bits) and the tag 2 * iteration + vote, written and read as one word.
__device__ __forceinline__ void st_slot(ulonglong2 *p, double v, unsigned long long tag) {
    asm volatile(
        "{\n\t.reg .b128 w;\n\tmov.b128 w, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], w;\n\t}"
        ::"l"(p), "l"(__double_as_longlong(v)), "l"(tag) : "memory");
}
__device__ __forceinline__ void ld_slot(const ulonglong2 *p, double &v, unsigned long long &tag) {
    long long b;
    asm volatile(
        "{\n\t.reg .b128 w;\n\tld.relaxed.gpu.global.b128 w, [%2];\n\tmov.b128 {%0, %1}, w;\n\t}"
        : "=l"(b), "=l"(tag) : "l"(p) : "memory");
    v = __longlong_as_double(b);
}

// One warp waits until slots [0, count) carry the iteration `iter`; a[j] is the value of slot
// lane + 32 j, *vote slot 0's vote.  Returns false when limit_ns passes first.
__device__ bool wait_slots(const ulonglong2 *slots, int count, unsigned long long iter,
                           double (&a)[kPartLoads], int *vote, long long limit_ns = kWaitLimitNs) {
    const int lane = threadIdx.x & 31;
    long long t0 = 0;
    for (unsigned spin = 0;; ++spin) {
        bool here = true;
        unsigned long long tag[kPartLoads];
#pragma unroll
        for (int j = 0; j < kPartLoads; ++j) {
            a[j] = 0.0;
            tag[j] = 2 * iter;
            if (lane + 32 * j < count) ld_slot(slots + lane + 32 * j, a[j], tag[j]);
            here = here && (tag[j] >> 1) == iter;
        }
        if (__all_sync(0xffffffffu, here)) {
            *vote = __shfl_sync(0xffffffffu, (int)(tag[0] & 1), 0);
            return true;
        }
        if ((spin & 63u) == 63u) {
            const long long now = global_timer_ns();
            if (t0 == 0) t0 = now;
            if (__any_sync(0xffffffffu, now - t0 > limit_ns)) return false;
        }
    }
}

// What the CTA's threads share.
template <typename T>
struct PersSmem {
    FoldSmem<2> fold;
    StepScalars<T> step;
    int vote, late;
};

// Sums over CTAs [0, ctas) of their first TT threads' v[k]: use(k, sum) runs in one thread of
// each CTA per quantity, and the other threads see what it wrote after the call.  Every CTA of
// the grid waits.  PUBLISH: the CTAs' earlier writes are visible to all after the exchange.
// meanwhile runs in every thread while the sums travel.  Returns false on a wait that ran out or
// CTA 0's vote to stop.
template <int NV, bool PUBLISH, typename T, typename F, typename M>
__device__ __forceinline__ bool exchange(const T (&v)[NV], int TT, int ctas,
                                         ulonglong2 *slots, unsigned long long iter, int my_vote,
                                         PersSmem<T> &sm, F &&use, M &&meanwhile) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const double s = fold_block<NV>(v, TT, sm.fold);
    ulonglong2 *mine = slots + (int64_t)warp * ctas;
    if (warp < NV && lane == 0 && (int)blockIdx.x < ctas) {
        if (PUBLISH) __threadfence();
        st_slot(mine + blockIdx.x, s, 2 * iter + my_vote);
    }
    meanwhile();
    if (warp < NV) {
        double a[kPartLoads];
        int vt = 0;
        const bool ok = wait_slots(mine, ctas, iter, a, &vt);
        if (PUBLISH) __threadfence();
        const double sum = sum_parts(a);
        if (lane == 0) {
            use(warp, sum);
            if (!ok) sm.late = 1;
            if (warp == 0) sm.vote = vt;
        }
    }
    __syncthreads();
    return sm.late == 0 && sm.vote == 0;
}

// All CTAs' earlier writes are visible to all CTAs after it.  Returns false on a wait that ran
// out.  `expected`: slots waited for (the grid's CTAs).
__device__ __forceinline__ bool grid_barrier(ulonglong2 *slots, int expected,
                                             unsigned long long iter, int *late,
                                             long long limit_ns = kWaitLimitNs) {
    __syncthreads();
    if (threadIdx.x < 32) {
        if (threadIdx.x == 0) {
            __threadfence();
            st_slot(slots + blockIdx.x, 0.0, 2 * iter);
        }
        double a[kPartLoads];
        int vote;
        if (!wait_slots(slots, expected, iter, a, &vote, limit_ns) && threadIdx.x == 0) *late = 1;
        __threadfence();
    }
    __syncthreads();
    return *late == 0;
}

// Slots of a solve: the p.q sums, the r.z and r.r sums, the barrier after the p update.
constexpr int kSlotsPq = 0;
constexpr int kSlotsR = 32 * kPartLoads;
constexpr int kSlotsP = 3 * 32 * kPartLoads;
constexpr int kSlotsTotal = 4 * 32 * kPartLoads;

template <typename T>
struct PersArgs {
    int32_t n, n_slices, width;  // width: stored entries of the widest slice
    const int64_t *sp;
    const T *val;
    T *x, *r, *p, *q;
    const T *dinv;
    T *zp;  // resident form with PAIRS: (D^-1 r, p) of every row
    IterGrid pq, sw;
    bool same;  // pq == sw
    IterKeep keep;
    ulonglong2 *slots;
    CgScalars *sc;
};

// Coherent load and store of a row's pair.
__device__ __forceinline__ void ld_pair(const double *p, double &z, double &v) {
    asm volatile("ld.global.ca.v2.f64 {%0,%1}, [%2];" : "=d"(z), "=d"(v) : "l"(p) : "memory");
}
__device__ __forceinline__ void ld_pair(const float *p, float &z, float &v) {
    asm volatile("ld.global.ca.v2.f32 {%0,%1}, [%2];" : "=f"(z), "=f"(v) : "l"(p) : "memory");
}
__device__ __forceinline__ void st_pair(double *p, double z, double v) {
    *reinterpret_cast<double2 *>(p) = make_double2(z, v);
}
__device__ __forceinline__ void st_pair(float *p, float z, float v) {
    *reinterpret_cast<float2 *>(p) = make_float2(z, v);
}

// RES: the resident form.  Otherwise vectors and matrix are streamed from L2 / HBM; `own` there
// says that each thread's product rows are its sweep rows (q needs no publishing).
template <typename T, int R, int L, typename ColT, int UU, bool RES, bool PAIRS, int THREADS, int CTAS = 1>
__global__ void __launch_bounds__(THREADS, CTAS)
cg_persistent(PersArgs<T> a, ColT col) {
    __shared__ PersSmem<T> sm;
    extern __shared__ __align__(16) unsigned char dyn[];
    const int t = threadIdx.x;
    const int32_t n = a.n;
    CgScalars *sc = a.sc;
    const uint64_t pol = policy_stream(a.keep.matrix), pol_v = policy_stream(a.keep.vectors);
    const long long t_start = global_timer_ns();
    const long long budget = sc->budget_ns;
    double rho = sc->rho;  // thread 0's is the current one
    T beta = T(0);
    const double limit = sc->tol2 * sc->bb;
    int iters = sc->iters;
    const int max_iter = sc->max_iter;
    int done = sc->done;
    if (t == 0) sm.late = sm.vote = 0;
    // the thread's slice-lanes g0, g0 + pq.threads, ... below g1 and vectors k0, ... below k1
    const int64_t g1 = t < a.pq.threads ? iter_end(a.pq.chunk, (int64_t)a.n_slices * L) : 0;
    const int64_t g0 = iter_begin(a.pq.chunk);
    const int64_t k1 =
        t < a.sw.threads ? iter_end(a.sw.chunk, ((int64_t)n + Vec16<T>::n - 1) / Vec16<T>::n) : 0;
    const int64_t k0 = iter_begin(a.sw.chunk);
    const bool own = R == Vec16<T>::n && a.same;

    // resident form: the lane's matrix rows in shared memory, entry u of all threads together
    struct alignas(sizeof(T) * R < 16 ? sizeof(T) * R : 16) ValVec { T e[R]; };
    struct alignas(R == 1 ? 4 : (R == 2 ? 8 : 16)) ColVec { int32_t e[R]; };
    ValVec *s_val = reinterpret_cast<ValVec *>(dyn);
    ColVec *s_col = reinterpret_cast<ColVec *>(s_val + (int64_t)a.width * blockDim.x);
    T x[R], r[R], p[R], d[R], z[R];
    int w = 0;
    const int64_t row0 = g0 * R;
    if constexpr (RES) {
        if (g0 < g1) {
            const SliceLane s = slice_open<R, L>(g0, a.sp, col);
            w = s.w;
            for (int u = 0; u < w; ++u) {
                ValVec v;
                ColVec c;
                ld_stream(a.val + s.at + (int64_t)u * (L * R), pol, v.e);
                col.template load<R>(s.at + (int64_t)u * (L * R), 0, pol, s.cbase, c.e);
                s_val[(int64_t)u * blockDim.x + t] = v;
                s_col[(int64_t)u * blockDim.x + t] = c;
            }
        }
#pragma unroll
        for (int i = 0; i < R; ++i) {
            const bool in = g0 < g1 && row0 + i < n;
            x[i] = in ? a.x[row0 + i] : T(0);
            r[i] = in ? a.r[row0 + i] : T(0);
            p[i] = in ? a.p[row0 + i] : T(0);
            d[i] = in ? a.dinv[row0 + i] : T(0);
            if (PAIRS) {  // the first product's beta p + D^-1 r is p
                if (in) st_pair(a.zp + 2 * (row0 + i), p[i], T(0));
                z[i] = p[i];
                p[i] = T(0);
            }
        }
    }
    __syncthreads();
    if (PAIRS && !done && !grid_barrier(a.slots + kSlotsP, (int)gridDim.x, 1, &sm.late)) done = 4;

    unsigned long long it = 0;
    while (!done) {
        ++it;
        // phase 1: q = A p, p.q
        T acc[R];
        T vt = T(0);
        if constexpr (RES) {
#pragma unroll
            for (int i = 0; i < R; ++i) acc[i] = T(0);
            for (int u0 = 0; u0 < w; u0 += UU) {
                ColVec c[UU];
                T xv[UU][R], zv[PAIRS ? UU : 1][R];
#pragma unroll
                for (int u = 0; u < UU; ++u) {
                    if (u0 + u < w) {
                        c[u] = s_col[(int64_t)(u0 + u) * blockDim.x + t];
                    } else {
#pragma unroll
                        for (int i = 0; i < R; ++i) c[u].e[i] = -1;
                    }
                }
#pragma unroll
                for (int u = 0; u < UU; ++u)
#pragma unroll
                    for (int i = 0; i < R; ++i) {
                        if constexpr (PAIRS) {
                            xv[u][i] = zv[u][i] = T(0);
                            if (c[u].e[i] >= 0)
                                ld_pair(a.zp + 2 * (int64_t)c[u].e[i], zv[u][i], xv[u][i]);
                        } else {
                            xv[u][i] = c[u].e[i] >= 0 ? ld_x_coherent(a.p + c[u].e[i]) : T(0);
                        }
                    }
#pragma unroll
                for (int u = 0; u < UU; ++u) {
                    if (PAIRS) {
#pragma unroll
                        for (int i = 0; i < R; ++i) xv[u][i] = fma_t(beta, xv[u][i], zv[u][i]);
                    }
                    if (u0 + u < w) {
                        const ValVec v = s_val[(int64_t)(u0 + u) * blockDim.x + t];
#pragma unroll
                        for (int i = 0; i < R; ++i)
                            if (c[u].e[i] >= 0) acc[i] = fma_t(v.e[i], xv[u][i], acc[i]);
                    }
                }
            }
#pragma unroll
            for (int i = 0; i < R; ++i) {
                if (PAIRS) p[i] = fma_t(beta, p[i], z[i]);
                if (g0 < g1 && row0 + i < n) vt = fma_t(p[i], acc[i], vt);
            }
        } else {
            for (int64_t g = g0; g < g1; g += a.pq.threads) {
                slice_rows<T, R, L, true, UU>(g / L, (int)(g % L), a.sp, col, a.val, a.p, pol,
                                              acc);
                store_rows<T, R>(a.q, g * R, n, acc);
#pragma unroll
                for (int i = 0; i < R; ++i)
                    if (g * R + i < n) vt = fma_t(a.p[g * R + i], acc[i], vt);
            }
        }
        const T v1[1] = {vt};
        // CTA 0's vote to stop on the wall-clock budget
        const int my_vote =
            blockIdx.x == 0 && budget > 0 && global_timer_ns() - t_start > budget ? 1 : 0;
        auto take_pq = [&](int, double pq) { step_alpha(rho, pq, sm.step); };
        const bool go = (RES || own) ? exchange<1, false>(v1, a.pq.threads, a.pq.ctas,
                                                          a.slots + kSlotsPq, it, my_vote, sm,
                                                          take_pq, [] {})
                                     : exchange<1, true>(v1, a.pq.threads, a.pq.ctas,
                                                         a.slots + kSlotsPq, it, my_vote, sm,
                                                         take_pq, [] {});
        if (!go) {
            done = 4;
            break;
        }
        if (sm.step.done) {
            done = 3;
            break;
        }
        // phase 2: x += alpha p, r -= alpha q, r.z, r.r
        const T alpha = sm.step.coef;
        T vz = T(0), vr = T(0);
        if constexpr (RES) {
#pragma unroll
            for (int i = 0; i < R; ++i) {
                if (g0 < g1 && row0 + i < n) {
                    r[i] = fma_t(-alpha, acc[i], r[i]);
                    z[i] = d[i] * r[i];
                    vz = fma_t(r[i], z[i], vz);
                    vr = fma_t(r[i], r[i], vr);
                    if (PAIRS) st_pair(a.zp + 2 * (row0 + i), z[i], p[i]);
                }
            }
        } else {
            sweep_update_xr<T, 1>(n, k0, k1, a.sw.threads, pol_v, alpha, a.x, a.r, a.p, a.q, a.dinv, vz, vr);
        }
        const T v2[2] = {vz, vr};
        ++iters;
        if (!exchange<2, PAIRS>(v2, a.sw.threads, a.sw.ctas, a.slots + kSlotsR, it, 0, sm,
                                [&](int k, double sum) {
                                    if (k == 0) {
                                        step_beta(rho, sum, sm.step);
                                        rho = sum;
                                    } else {
                                        sm.step.rr = sum;
                                        sm.step.done = step_done(sum, limit, iters, max_iter);
                                    }
                                },
                                [&] {  // nothing waits for x
                                    if constexpr (RES) {
#pragma unroll
                                        for (int i = 0; i < R; ++i)
                                            x[i] = fma_t(alpha, p[i], x[i]);
                                    }
                                })) {
            done = 4;
            break;
        }
        beta = sm.step.coef;
        done = sm.step.done;
        if (done) {
            if (blockIdx.x == 0 && t == 0) sc->rr = sm.step.rr;
            break;
        }
        // phase 3: p = D^-1 r + beta p
        if constexpr (PAIRS) continue;
        if constexpr (RES) {
#pragma unroll
            for (int i = 0; i < R; ++i) p[i] = fma_t(beta, p[i], z[i]);
            if (g0 < g1) store_rows<T, R>(a.p, row0, n, p);
        } else {
            sweep_update_p<T, 1>(n, k0, k1, a.sw.threads, pol_v, beta, a.r, a.dinv, a.p);
        }
        if (!grid_barrier(a.slots + kSlotsP, (int)gridDim.x, it, &sm.late)) {
            done = 4;
            break;
        }
    }
    if constexpr (RES) {
        if (g0 < g1) store_rows<T, R>(a.x, row0, n, x);
    }
    if (t == 0) {
        if (done == 4) atomicExch(&sc->done, 4);
        else if (blockIdx.x == 0) atomicCAS(&sc->done, 0, done);
        if (blockIdx.x == 0) {
            sc->iters = iters;
            sc->rho = rho;
            sc->beta = (double)beta;
        }
    }
}

// Diagnostic: a barrier that expects one CTA more than the grid has, so no wait can ever be
// released -- every CTA must leave through the time limit and record done = 4.
__global__ void barrier_timeout_probe(CgScalars *sc, ulonglong2 *slots, long long limit_ns) {
    __shared__ int late;
    if (threadIdx.x == 0) late = 0;
    if (!grid_barrier(slots, gridDim.x + 1, 1, &late, limit_ns) && threadIdx.x == 0)
        atomicExch(&sc->done, 4);
}

}  // namespace

spmv_status_t diag_barrier_timeout(int ctas, double limit_s, int *done_out, cudaStream_t st) {
    // one slot more than there are CTAs stays empty
    const size_t slots_at = (sizeof(CgScalars) + 255) / 256 * 256;
    const size_t bytes = slots_at + sizeof(ulonglong2) * ((size_t)ctas + 1);
    unsigned char *mem = nullptr;
    // the wait reads at most 32 kPartLoads slots, so the empty one must be among them
    ctas = std::min(ctas, 32 * kPartLoads - 1);
    GB_CUDA(gb_malloc_async((void **)&mem, bytes, st));
    spmv_status_t s = cuda_status(cudaMemsetAsync(mem, 0, bytes, st));
    CgScalars *sc = (CgScalars *)mem;
    ulonglong2 *slots = (ulonglong2 *)(mem + slots_at);
    long long limit_ns = (long long)(limit_s * 1e9);
    void *args[] = {&sc, &slots, &limit_ns};
    if (s == SPMV_OK)
        s = cuda_status(cudaLaunchCooperativeKernel((const void *)barrier_timeout_probe,
                                                    dim3(ctas), dim3(32), args, 0, st));
    CgScalars h{};
    if (s == SPMV_OK)
        s = cuda_status(cudaMemcpyAsync(&h, sc, sizeof(CgScalars), cudaMemcpyDeviceToHost, st));
    if (s == SPMV_OK) s = cuda_status(cudaStreamSynchronize(st));
    cudaFreeAsync(mem, st);
    cudaStreamSynchronize(st);
    *done_out = h.done;
    return s;
}

static DevBuf<double> &pair_buffer(CgWork &w, double) { return w.zp; }
static DevBuf<float> &pair_buffer(CgWork &w, float) { return w.zp32; }

// One cooperative launch running the recurrence to its end; FP64 (outer scalars, FP64 work
// vectors) or FP32 (inner scalars of the refinement, FP32 work vectors and values).
template <typename T>
static spmv_status_t run_persistent(spmv_matrix_t A, PersArgs<T> a, const cg_options_t &o,
                                    CgScalars *out, cudaStream_t st) {
    CgWork &w = A->cg;
    constexpr bool f32 = sizeof(T) == 4;
    a.n = A->n;
    a.n_slices = A->n_slices;
    a.width = A->max_width;
    a.sp = A->slice_ptr.p;
    a.sc = (CgScalars *)w.scal.p + (f32 ? 1 : 0);
    a.sw = cg_sweep_grid(A, Vec16<T>::n);
    a.keep = cg_keep(A, (int)sizeof(T));
    if (!w.slots.p) GB_TRY(w.slots.alloc(kSlotsTotal, &A->bytes));
    a.slots = w.slots.p;
    GB_CUDA(cudaMemsetAsync(w.slots.p, 0, sizeof(ulonglong2) * kSlotsTotal, st));
    const long long budget = o.timeout_s > 0 ? (long long)(o.timeout_s * 1e9) : 0;
    GB_CUDA(cudaMemcpyAsync(&a.sc->budget_ns, &budget, sizeof(budget), cudaMemcpyHostToDevice,
                            st));
    auto launch = [&](auto cols) -> spmv_status_t {
        using ColT = decltype(cols);
        return with_shape<T>(A->S, [&](auto rt, auto lt) -> spmv_status_t {
            constexpr int R = decltype(rt)::value, L = decltype(lt)::value;
            constexpr int UU = pq_unroll((int)sizeof(T) * R);
            a.pq = cg_pq_grid(A, L, (int)sizeof(T) * R);
            a.same = a.pq == a.sw;
            const int ctas = std::max(a.pq.ctas, a.sw.ctas);
            const int threads = std::max(a.pq.threads, a.sw.threads);
            size_t smem = 0;
            const void *kern = nullptr;
            if constexpr (R == Vec16<T>::n) {
                // resident form: one slice-lane per thread, the matrix within shared memory
                const size_t need = (size_t)A->max_width * threads * R * (sizeof(T) + 4);
                const size_t room = device_facts().max_smem_optin - sizeof(PersSmem<T>) - 1024;
                if (a.same && a.pq.single() && need <= room) {
                    const bool pairs = threads <= 512;
                    // CTAs of up to 128 threads take the registers of five entries in flight
                    // (up to 128 a thread); larger ones three at 64 registers, so that the SMs hold the
                    // kernels of several streams: solves/s of 1 / 4 / 16 host threads, five and
                    // three: 48K rows 435 / 835 / 894 and 431 / 1,273 / 1,480, 118K rows 261 / 303
                    // / 300 and 270 / 467 / 464 (256-thread CTAs that streamed the matrix: 243 /
                    // 850 / 1,099 and 185 / 322 / 430)
                    kern = pairs && threads <= 128
                               ? (const void *)cg_persistent<T, R, L, ColT, 5, true, true, 512>
                           : pairs
                               ? (const void *)cg_persistent<T, R, L, ColT, 3, true, true, 512, 2>
                               : (const void *)cg_persistent<T, R, L, ColT, 5, true, false, 1024>;
                    if (pairs) {
                        DevBuf<T> &zp = pair_buffer(w, T{});
                        if (!zp.p) GB_TRY(zp.alloc(2 * (size_t)A->n, &A->bytes));
                        a.zp = zp.p;
                    }
                    smem = need;
                    // the same value whatever this handle needs: it is the function's, shared by
                    // all handles and host threads
                    GB_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                 (int)room));
                }
            }
            if (!kern)
                kern = cg_pq_deep(A, UU)
                           ? (const void *)cg_persistent<T, R, L, ColT, UU, false, false, 1024>
                           : (const void *)cg_persistent<T, R, L, ColT, 2, false, false, 1024>;
            int per_sm = 0;
            GB_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem));
            if (per_sm < 1) return SPMV_ERR_UNSUPPORTED;
            void *args[] = {&a, &cols};
            GB_CUDA(cudaLaunchCooperativeKernel(kern, dim3(ctas), dim3(threads), args, smem, st));
            GB_CUDA(cudaMemcpyAsync(w.h_scal, w.scal.p, 2 * sizeof(CgScalars),
                                    cudaMemcpyDeviceToHost, st));
            GB_CUDA(cudaStreamSynchronize(st));
            *out = w.h_scal[f32 ? 1 : 0];
            return SPMV_OK;
        });
    };
    if (A->index_bits == 16) return launch(Cols16{A->sell_col16.p, A->col_start.p});
    return launch(Cols32{A->sell_col.p});
}

spmv_status_t cg_persistent64(spmv_matrix_t A, const cg_options_t &o, CgScalars *out,
                              cudaStream_t st) {
    CgWork &w = A->cg;
    PersArgs<double> a{};
    a.val = A->sell_val.p;
    a.x = w.x.p, a.r = w.r.p, a.p = w.p.p, a.q = w.q.p, a.dinv = w.dinv.p;
    return run_persistent<double>(A, a, o, out, st);
}

spmv_status_t cg_persistent32(spmv_matrix_t A, const cg_options_t &o, CgScalars *out,
                              cudaStream_t st) {
    CgWork &w = A->cg;
    PersArgs<float> a{};
    a.val = A->sell_val32.p;
    a.x = w.d32.p, a.r = w.r32.p, a.p = w.p32.p, a.q = w.q32.p, a.dinv = w.dinv32.p;
    return run_persistent<float>(A, a, o, out, st);
}

}  // namespace gb
