// spmv.cu -- SpMV kernels (the multi-vector products are in spmm.cu).
//
// spmv_sell_thin<T, R, L>: L lanes per slice of S = L R rows, lane l owns rows l R .. l R + R - 1
//   of the slice (one or two).  Because a slice is stored column-major (Sec. 4.2), step t of the
//   lanes reads S consecutive values and column indices: one R-wide vector load per lane, fully
//   coalesced, streamed evict-first so the matrix never displaces x from L2.  x is gathered
//   through the read-only L1 path; with a banded (Cuthill-McKee) order the gathers of
//   neighbouring rows hit the same lines (Sec. 4.3, 5.1).  Each row accumulates its entries
//   in ascending column order with fused multiply-add from +0.0; padding entries (column -1)
//   are skipped.  Column indices come as int32 or (when every slice spans fewer than 65,535
//   columns) as 16-bit offsets from the slice's col_start (Sec. 5.1), 10 instead of 12 bytes
//   per FP64 non-zero.  Matrices up to a few million rows (use_thin).
// spmv_sell_gs / spmv_sell_occ: larger matrices, one or two rows per lane in FP64 and four in FP32;
//   a grid of four CTAs per SM striding over the slice-lanes with five entries of each row in
//   flight, or (FP64) one slice-lane per thread at 32 registers; the one whose widest slice needs
//   fewer dependent load rounds is launched.  spmv_sell: FP64 at four or eight rows per lane.
// spmv_csr: the naive baseline of Sec. 4.3, thread per CSR row.
#include <type_traits>

#include "common.cuh"
#include "ptx.cuh"

namespace gb {
namespace {

// Hint: bring bytes (a multiple of 16) from p (16-byte aligned) on into L2.
__device__ __forceinline__ void prefetch_l2_bulk(const void *p, uint32_t bytes) {
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes));
}
// 8 bytes from global to shared memory, not waited for.
__device__ __forceinline__ void copy_async8(volatile void *to, const void *from) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(
                     (uint32_t)__cvta_generic_to_shared((const void *)to)), "l"(from));
}

// y = A x, or with AXPBY y = alpha (A x) + beta y evaluated as fma(alpha, t, beta y) (y is not
// read when beta == 0), t being the row sum in column order.
// gt: the slice-lane this thread computes (slice gt / L, lane gt % L).  The entries of a row
// go in blocks of U (all loads of a block issued before its gathers, and those before its
// FMAs), the rest one at a time.
template <typename T, int R, int L, int U, typename ColT, bool AXPBY>
__device__ __forceinline__ void spmv_sell_body(int64_t gt, int32_t n, int32_t n_slices,
                                               const int64_t *__restrict__ sp, ColT cols,
                                               const T *__restrict__ val,
                                               const T *x, T *y,
                                               T alpha, T beta) {
    // L lanes per slice, R rows per lane: S = L R rows per slice
    constexpr int S = L * R;
    const int64_t slice = gt / L;
    const int lane = (int)(gt % L);
    if (slice >= n_slices) return;
    const int64_t base = sp[slice];
    const int w = (int)((sp[slice + 1] - base) / S);
    const int32_t cbase = cols.base(slice);
    const T *vp = val + base + lane * R;
    const int64_t cat = base + lane * R;
    const uint64_t pol = policy_evict_first();
    T acc[R];
#pragma unroll
    for (int i = 0; i < R; ++i) acc[i] = T(0);
    int t = 0;
    for (; t + U <= w; t += U) {
        T v[U][R];
        int32_t c[U][R];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            ld_stream(vp + (int64_t)(t + u) * S, pol, v[u]);
            cols.template load<R>(cat + (int64_t)(t + u) * S, slice, pol, cbase, c[u]);
        }
        T xv[U][R];
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int i = 0; i < R; ++i) xv[u][i] = c[u][i] >= 0 ? ld_x(x + c[u][i]) : T(0);
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int i = 0; i < R; ++i)
                if (c[u][i] >= 0) acc[i] = fma_t(v[u][i], xv[u][i], acc[i]);
    }
    for (; t < w; ++t) {
        T v[R];
        int32_t c[R];
        ld_stream(vp + (int64_t)t * S, pol, v);
        cols.template load<R>(cat + (int64_t)t * S, slice, pol, cbase, c);
#pragma unroll
        for (int i = 0; i < R; ++i)
            if (c[i] >= 0) acc[i] = fma_t(v[i], ld_x(x + c[i]), acc[i]);
    }
    const int64_t row0 = slice * S + (int64_t)lane * R;
    if constexpr (AXPBY) {
#pragma unroll
        for (int i = 0; i < R; ++i) {
            if (row0 + i < n)
                acc[i] = beta != T(0) ? fma_t(alpha, acc[i], beta * y[row0 + i]) : alpha * acc[i];
        }
    }
    store_rows<T, R>(y, row0, n, acc);
}

template <typename T, int R, int L, int U, typename ColT, bool AXPBY>
__global__ void __launch_bounds__(1024)
spmv_sell(int32_t n, int32_t n_slices, const int64_t *__restrict__ sp, ColT cols,
          const T *__restrict__ val, const T *x, T *y, T alpha,
          T beta) {
    dep_wait();
    dep_allow();
    spmv_sell_body<T, R, L, U, ColT, AXPBY>((int64_t)blockIdx.x * blockDim.x + threadIdx.x, n,
                                            n_slices, sp, cols, val, x, y, alpha, beta);
}

// FP64 with one or two rows per lane, capped at 32 registers (2 x 1024 threads per SM), four
// entries in flight: for matrices whose widest slice needs fewer load rounds in blocks of four
// than of five (see go_sell).
template <typename T, int R, int L, int U, typename ColT, bool AXPBY>
__global__ void __launch_bounds__(1024, 2)
spmv_sell_occ(int32_t n, int32_t n_slices, const int64_t *__restrict__ sp, ColT cols,
              const T *__restrict__ val, const T *x, T *y, T alpha,
              T beta) {
    dep_wait();
    dep_allow();
    spmv_sell_body<T, R, L, U, ColT, AXPBY>((int64_t)blockIdx.x * blockDim.x + threadIdx.x, n,
                                            n_slices, sp, cols, val, x, y, alpha, beta);
}

// One or two rows per lane (FP32 four): a grid of at most kGsCtasPerSm 256-thread CTAs per SM
// strides over the slice-lanes, each thread keeping U = 5 entries of its rows in flight (a
// whole row of the tetrahedral meshes) at 64 registers.  Measured on the 6M-row mesh (S = 64):
// 66.3 us, against 69.6 us for one slice-lane per thread at 32 registers and 2,048 threads per
// SM (four entries in flight), 77.1 us with four entries and 68.3 us with two at six CTAs.  A
// dependent launch, as are the other two: 68.1 -> 66.3 us in a stream of products with the wait
// first thing in the kernel; behind the first requests for entries it cost 69.6.  AHEAD (a matrix of
// more than twice the L2): 66.3 -> 62.9 us, the 396 MB that the product cannot do without at 93 % of
// the copy rate; where the product before leaves a good part of the matrix in L2 it costs more than
// it saves (3.7M rows 39.7 -> 41.3).
constexpr int kGsBlock = 256;
constexpr int kGsCtasPerSm = 4;
template <typename T, int R, int L, int U, typename ColT, bool AXPBY, bool AHEAD>
__global__ void __launch_bounds__(kGsBlock, kGsCtasPerSm)
spmv_sell_gs(int32_t n, int32_t n_slices, const int64_t *__restrict__ sp, ColT cols,
             const T *__restrict__ val, const T *x, T *y, T alpha,
             T beta) {
    dep_wait();
    dep_allow();
    const int64_t items = (int64_t)n_slices * L;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    // AHEAD: thread 0 brings the entries of the CTA's next step into L2 in two bulk requests.  Their
    // bounds come a step earlier into shared memory, so that no register holds them.
    __shared__ volatile int64_t bound[2];
    bool first = true;
    for (int64_t gt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; gt < items; gt += stride) {
        if (AHEAD && threadIdx.x == 0) {
            if (!first) {
                asm volatile("cp.async.wait_all;");
                const int64_t e0 = bound[0], count = bound[1] - e0;
                if (gt + stride < items && count > 0 && count <= 65536) {
                    prefetch_l2_bulk(val + e0, (uint32_t)count * (uint32_t)sizeof(T));
                    prefetch_l2_bulk(cols.col + e0, (uint32_t)count * (uint32_t)sizeof(cols.col[0]));
                }
            }
            first = false;
            const int64_t s0 = (gt + 2 * stride) / L;
            if (s0 < n_slices) {
                const int64_t s1 = s0 + kGsBlock / L < n_slices ? s0 + kGsBlock / L : n_slices;
                copy_async8(&bound[0], sp + s0);
                copy_async8(&bound[1], sp + s1);
            }
        }
        spmv_sell_body<T, R, L, U, ColT, AXPBY>(gt, n, n_slices, sp, cols, val, x, y, alpha, beta);
    }
}

// One or two rows per lane, S / R lanes per slice (a slice may span several warps), U entries in
// flight, and the remainder of a row as one more round with the missing entries masked instead of
// one dependent round per entry.  A row is a chain of three or four dependent loads of 0.6 us, so
// below a few million rows time goes by how many waves of threads an SM takes and how many rounds
// a row takes: CTAS (CTAs of kThinBlock per SM) sets the registers, 64, 40 or 32, and with them
// the 1,024, 1,536 or 2,048 threads that an SM holds (see go_thin).  A dependent launch: slices
// and the first round of entries are requested while the kernel before still runs.  Measured (us,
// against four rows per lane, plain launches and registers as they fell): FP64 48K tetrahedra 3.4
// -> 2.0, 304K 5.9 -> 4.2, 1.3M 18.7 -> 13.7, 398K mixed-mesh rows 16 -> 11.7; FP32 304K 8 -> 2.4,
// 1.3M 10.8 -> 7.1, 6M 36 -> 32, 398K mixed 16.6 -> 5.9.  Same order and bits as spmv_sell.
constexpr int kThinBlock = 128;
template <typename T, int R, int L, int U, int CTAS, typename ColT, bool AXPBY>
__global__ void __launch_bounds__(kThinBlock, CTAS)
spmv_sell_thin(int32_t n, int32_t n_slices, const int64_t *__restrict__ sp, ColT cols,
               const T *__restrict__ val, const T *x, T *y, T alpha,
               T beta, bool add) {
    constexpr int S = L * R;
    const int64_t gt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t slice = gt / L;
    if (slice >= n_slices) {
        dep_wait();
        return;
    }
    const int lane = (int)(gt % L);
    const int64_t base = sp[slice];
    const int w = (int)((sp[slice + 1] - base) / S);
    const int32_t cbase = cols.base(slice);
    const int64_t at = base + lane * R;
    const uint64_t pol = policy_evict_first();
    T acc[R];
#pragma unroll
    for (int i = 0; i < R; ++i) acc[i] = T(0);
    T v[U][R];
    int32_t c[U][R];
    auto load = [&](int t, auto masked) {
        constexpr bool kMasked = decltype(masked)::value;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (!kMasked || t + u < w) {
                ld_stream(val + at + (int64_t)(t + u) * S, pol, v[u]);
                cols.template load<R>(at + (int64_t)(t + u) * S, slice, pol, cbase, c[u]);
            } else {
#pragma unroll
                for (int i = 0; i < R; ++i) {
                    v[u][i] = T(0);
                    c[u][i] = -1;
                }
            }
        }
    };
    auto multiply = [&] {
        T xv[U][R];
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int i = 0; i < R; ++i) xv[u][i] = c[u][i] >= 0 ? ld_x(x + c[u][i]) : T(0);
#pragma unroll
        for (int u = 0; u < U; ++u)
#pragma unroll
            for (int i = 0; i < R; ++i)
                if (c[u][i] >= 0) acc[i] = fma_t(v[u][i], xv[u][i], acc[i]);
    };
    // the matrix does not depend on the kernel before: its first entries are requested while that
    // one ends
    if (U <= w) load(0, std::false_type{});
    else load(0, std::true_type{});
    dep_wait();
    dep_allow();
    const int64_t row0 = gt * R;
    // y of the rows: in FP32 with the first gathers (0.2 us of a small product); in FP64, where the
    // registers are short, at the end (1.3M rows 20.8 against 26.0 us).  `add` is beta != 0: the
    // comparison in FP64 costs as much of the FP64 pipe as a multiply-add
    T y0[AXPBY ? R : 1];
    auto load_y = [&] {
#pragma unroll
        for (int i = 0; i < R; ++i) y0[i] = add && row0 + i < n ? y[row0 + i] : T(0);
    };
    if constexpr (AXPBY && sizeof(T) == 4) load_y();
    multiply();
    int t = U;
    for (; t + U <= w; t += U) {
        load(t, std::false_type{});
        multiply();
    }
    if (t < w) {
        load(t, std::true_type{});
        multiply();
    }
    if constexpr (AXPBY) {
        if constexpr (sizeof(T) == 8) load_y();
#pragma unroll
        for (int i = 0; i < R; ++i)
            acc[i] = add ? fma_t(alpha, acc[i], beta * y0[i]) : alpha * acc[i];
    }
    store_rows<T, R>(y, row0, n, acc);
}

// naive CSR baseline (Sec. 4.3): the column index is read first, then x[col] from global
// memory, thread per row
template <typename T>
__global__ void __launch_bounds__(256)
spmv_csr(int32_t n, const int32_t *__restrict__ rp, const int32_t *__restrict__ ci,
         const T *__restrict__ val, const T *__restrict__ x, T *__restrict__ y) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    T acc = T(0);
    for (int32_t k = rp[i]; k < rp[i + 1]; ++k) acc = fma_t(val[k], x[ci[k]], acc);
    y[i] = acc;
}

template <typename T>
__global__ void permute_kernel(int32_t n, int direction, const int32_t *__restrict__ perm,
                               const T *__restrict__ in, T *__restrict__ out) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (direction == 0) out[i] = in[perm[i]];
    else out[perm[i]] = in[i];
}

inline unsigned grid_for(int64_t threads, int block) {
    int64_t b = (threads + block - 1) / block;
    return (unsigned)(b < 1 ? 1 : b);
}

// A matrix of which a product leaves nothing in L2 for the next one.
template <typename T>
bool beyond_l2(const spmv_matrix_t A) {
    return (double)A->sell_entries * (sizeof(T) + A->index_bits / 8) >
           2.0 * device_facts().l2_bytes;
}

// Whether the strided form of FP64 rows at one or two per lane is spmv_sell_gs (else _occ).
bool strided_rows(const spmv_matrix_t A) {
    return load_rounds(A->max_width, 5) < load_rounds(A->max_width, 4);
}

// The products of larger matrices; (R, L) per slice height: lanes read 8 R bytes of values per
// entry in FP64 (16 B at S = 64, 32 B at S = 128), 16 in FP32.
template <typename T, int R, int L, int U, bool AXPBY>
spmv_status_t go_sell(spmv_matrix_t A, const T *val, const T *x, T *y, T alpha, T beta,
                      cudaStream_t st) {
    const int block = A->block;
    const unsigned grid = grid_for((int64_t)A->n_slices * L, block);
    auto strided = [&](auto c, auto aheadt) -> spmv_status_t {
        const int64_t cap = (int64_t)device_facts().sm_count * kGsCtasPerSm;
        const unsigned want = grid_for((int64_t)A->n_slices * L, kGsBlock);
        return launch_dependent(spmv_sell_gs<T, R, L, 5, decltype(c), AXPBY, decltype(aheadt)::value>,
                                (int64_t)want < cap ? want : (unsigned)cap, kGsBlock, st, A->n,
                                A->n_slices, A->slice_ptr.p, c, val, x, y, alpha, beta);
    };
    auto go = [&](auto c) -> spmv_status_t {
        using ColT = decltype(c);
        if constexpr (sizeof(T) == 4) {  // (ahead, 10.4M rows: 61.7 us cold and 61.3 in a row, without 60.9 and 62.0)
            return strided(c, std::false_type{});
        } else if constexpr (R <= 2) {
            if (strided_rows(A)) {
                // (not where x is gathered from all over: the entries then drive x out of L2, 6M rows
                // in random order 111 -> 130 us)
                const bool ahead = beyond_l2<T>(A) && (double)A->max_span * sizeof(T) <
                                                          device_facts().l2_bytes / 16.0;
                return ahead ? strided(c, std::true_type{}) : strided(c, std::false_type{});
            }
            return launch_dependent(spmv_sell_occ<T, R, L, U, ColT, AXPBY>, grid, block, st, A->n,
                                    A->n_slices, A->slice_ptr.p, c, val, x, y, alpha, beta);
        } else {
            return launch_dependent(spmv_sell<T, R, L, U, ColT, AXPBY>, grid, block, st, A->n,
                                    A->n_slices, A->slice_ptr.p, c, val, x, y, alpha, beta);
        }
    };
    if (A->index_bits == 16) return go(Cols16{A->sell_col16.p, A->col_start.p});
    return go(Cols32{A->sell_col.p});
}

// Products that spmv_sell_thin takes, unless the tuner has picked a form for the handle.  Products
// in a row (us, spmv_sell_gs or _occ / thin): FP64 rows of up to six entries in Cuthill-McKee
// order 304K 4.5 / 4.2, 796K 10.5 / 8.7, 3.1M 33.4 / 29.9, 6M 66.3 / 71.1; of two entries (a
// gradient's faces) 600K 5.3 / 4.5, 2.6M 22.6 / 17.2; longer rows 647K 20.8 / 17.1, 1.8M 44.6 /
// 43.5, 3M 70.8 / 69.9 but with alpha and beta 82.6 / 84.5.  FP32: 3.1M 17.7 / 17.0, 6M 33.5 /
// 32.4, and beyond the L2, 10.4M, 62.0 / 64.7; longer rows 1.8M 27.6 / 23.8.  With nothing in the
// caches the line lies lower, since thin's CTAs come and go with their chains of loads (FP64 1.3M
// 21.9 / 21.9, 3.1M 37.9 / 39.9, FP32 6M 38.7 / 40.7): that is the tuner's to find.
template <typename T>
bool use_thin(const spmv_matrix_t A) {
    constexpr bool f32 = sizeof(T) == 4;
    if (A->spmv_form[f32]) return A->spmv_form[f32] == kFormThin;
    const bool longer = A->max_width > 2 && A->mean_width > 6.f;
    if (f32) return longer || A->max_width <= 2 || !beyond_l2<T>(A);
    return A->n <= (longer ? 2000000 : 3500000);
}

// Rows per lane, entries in flight and registers of spmv_sell_thin, by the threads that an SM
// then has to run.
template <typename T, bool AXPBY>
spmv_status_t go_thin(spmv_matrix_t A, const T *val, const T *x, T *y, T alpha, T beta,
                      cudaStream_t st) {
    using std::integral_constant;
    auto launch = [&](auto rt, auto ut, auto ct, auto heightt) -> spmv_status_t {
        constexpr int R = decltype(rt)::value, U = decltype(ut)::value;
        constexpr int CTAS = decltype(ct)::value, L = decltype(heightt)::value / R;
        const int block = A->block < kThinBlock ? A->block : kThinBlock;
        const unsigned grid = grid_for((int64_t)A->n_slices * L, block);
        if (A->index_bits == 16)
            return launch_dependent(spmv_sell_thin<T, R, L, U, CTAS, Cols16, AXPBY>, grid, block,
                                    st, A->n, A->n_slices, A->slice_ptr.p,
                                    Cols16{A->sell_col16.p, A->col_start.p}, val, x, y, alpha,
                                    beta, beta != T(0));
        return launch_dependent(spmv_sell_thin<T, R, L, U, CTAS, Cols32, AXPBY>, grid, block, st,
                                A->n, A->n_slices, A->slice_ptr.p, Cols32{A->sell_col.p}, val, x,
                                y, alpha, beta, beta != T(0));
    };
    auto go = [&](auto rt, auto ut, auto ct) -> spmv_status_t {
        switch (A->S) {
            case 32: return launch(rt, ut, ct, integral_constant<int, 32>{});
            case 64: return launch(rt, ut, ct, integral_constant<int, 64>{});
            case 128: return launch(rt, ut, ct, integral_constant<int, 128>{});
            case 256: return launch(rt, ut, ct, integral_constant<int, 256>{});
        }
        return SPMV_ERR_INVALID_ARG;
    };
    constexpr bool f32 = sizeof(T) == 4;
    constexpr integral_constant<int, 1> one{};
    constexpr integral_constant<int, 2> two{};
    constexpr integral_constant<int, 5> u5{};
    constexpr integral_constant<int, 6> u6{};
    constexpr integral_constant<int, 7> u7{};
    constexpr integral_constant<int, 8> regs64{};
    constexpr integral_constant<int, 12> regs40{};
    constexpr integral_constant<int, 16> regs32{};
    // The entries in flight are a whole row of the tetrahedral meshes (5), two for two-entry rows
    // (five, four masked: 600K rows 6.8 against 4.5 us), and for longer rows what the registers
    // hold: FP64 6 (4: 192K mixed-mesh rows 8.0 against 6.5 us, 7: 7.2), FP32 7 (5: 292K rows 5.2
    // against 4.2).
    const bool narrow = A->max_width <= 2;
    const bool longer = !narrow && A->mean_width > 6.f;
    auto threads_per_sm = [&](int R) {
        return (int64_t)A->n_slices * (A->S / R) / device_facts().sm_count;
    };
    // Two rows per lane halve the threads where one would need more than the SM holds in a single
    // wave: FP32 (304K rows 3.9 against 2.4 us; 192K mixed 3.2 against 4.1, 222K even), and
    // two-entry rows.  Other FP64 rows have no registers for two (304K rows 7.0 against 4.9).
    const bool two_rows = narrow || (f32 && (longer ? threads_per_sm(1) > 1280
                                                    : A->n > 256 * 1024));
    const int64_t threads = threads_per_sm(two_rows ? 2 : 1);
    // 64 registers for up to 1,024 threads; else those that let one wave of 1,536 or 2,048 threads
    // cover the rows (FP64 162K rows: 3.3 us at 40 registers, 4.0 at 32; 304K rows, 2,000 threads:
    // 4.4 and 4.2; FP32 511K rows, 1,680 threads: 3.9 and 3.5).  With more waves two rows per lane
    // do better at 40 (878K two-entry rows 6.3, against 7.6 at 32), one row at 32 (1M rows 10.8,
    // against 11.1 at 40 and 13.7 at 64)
    const bool one_wave32 = threads > 1536 && threads <= 2048;
    if (narrow) {
        if (threads <= 1024) return go(two, two, regs64);
        return one_wave32 ? go(two, two, regs32) : go(two, two, regs40);
    }
    if constexpr (f32) {
        if (!two_rows) return longer ? go(one, u7, regs64) : go(one, u5, regs64);
        if (longer) {  // 398K mixed 5.1 at 40 registers, 5.9 at 64; 942K 14.1 at 64 (U = 7: 14.4)
            if (threads <= 1024) return go(two, u7, regs64);
            return threads <= 1536 ? go(two, u7, regs40) : go(two, u6, regs64);
        }
        if (threads <= 1024) return go(two, u5, regs64);
        return one_wave32 ? go(two, u5, regs32) : go(two, u5, regs40);
    } else {
        if (longer) return go(one, u6, regs64);
        // rows whose gathers miss L1 (random cell order) are bound by the loads in flight: 1.3M
        // rows 25.6 at 64 registers, 27.7 at 32
        if (threads <= 1024 || (A->max_span > 65535 && A->n > 1000000))
            return go(one, u5, regs64);
        // y = alpha A x + beta y spills at 32 (1.3M rows 20.8 against 29.0)
        return AXPBY || threads <= 1536 ? go(one, u5, regs40) : go(one, u5, regs32);
    }
}

template <typename T, bool AXPBY = false>
spmv_status_t launch_sell(spmv_matrix_t A, const T *val, const T *x, T *y, T alpha = T(1),
                          T beta = T(0), cudaStream_t st = nullptr) {
    if (A->n == 0) return SPMV_OK;
    if (use_thin<T>(A)) return go_thin<T, AXPBY>(A, val, x, y, alpha, beta, st);
    if constexpr (sizeof(T) == 8) {
        switch (A->S) {
            case 32: return go_sell<T, 1, 32, 4, AXPBY>(A, val, x, y, alpha, beta, st);
            case 64: return go_sell<T, 2, 32, 4, AXPBY>(A, val, x, y, alpha, beta, st);
            case 128: return go_sell<T, 4, 32, 2, AXPBY>(A, val, x, y, alpha, beta, st);
            case 256: return go_sell<T, 8, 32, 1, AXPBY>(A, val, x, y, alpha, beta, st);
        }
    } else {
        switch (A->S) {
            case 32: return go_sell<T, 4, 8, 5, AXPBY>(A, val, x, y, alpha, beta, st);
            case 64: return go_sell<T, 4, 16, 5, AXPBY>(A, val, x, y, alpha, beta, st);
            case 128: return go_sell<T, 4, 32, 5, AXPBY>(A, val, x, y, alpha, beta, st);
            case 256: return go_sell<T, 4, 64, 5, AXPBY>(A, val, x, y, alpha, beta, st);
        }
    }
    return SPMV_ERR_INVALID_ARG;
}

}  // namespace

bool product_is_thin(const spmv_matrix_t A, bool f32) {
    return f32 ? use_thin<float>(A) : use_thin<double>(A);
}

// CTA size of the product (the handle's first precision); A->block where the kernel leaves it open.
int product_block(const spmv_matrix_t A) {
    const bool f32 = !A->has64();
    if (A->variant != SPMV_VARIANT_SELL) return A->block;
    if (product_is_thin(A, f32)) return A->block < kThinBlock ? A->block : kThinBlock;
    return f32 || (A->S <= 64 && strided_rows(A)) ? kGsBlock : A->block;
}

spmv_status_t launch_spmv64(spmv_matrix_t A, const double *x, double *y, cudaStream_t st) {
    if (A->variant == SPMV_VARIANT_CSR) return launch_spmv_csr64(A, x, y, st);
    if (A->variant == SPMV_VARIANT_SELL_WINDOW) return launch_window64(A, x, y, st);
    if (A->variant == SPMV_VARIANT_SELL_BULK) {
        bool launched = false;
        GB_TRY(launch_bulk64(A, x, y, st, &launched));
        if (launched) return SPMV_OK;
    }
    return launch_sell<double>(A, A->sell_val.p, x, y, 1.0, 0.0, st);
}

spmv_status_t launch_axpby64(spmv_matrix_t A, double alpha, const double *x, double beta,
                             double *y, cudaStream_t st) {
    return launch_sell<double, true>(A, A->sell_val.p, x, y, alpha, beta, st);
}

spmv_status_t launch_axpby32(spmv_matrix_t A, float alpha, const float *x, float beta, float *y,
                             cudaStream_t st) {
    return launch_sell<float, true>(A, A->sell_val32.p, x, y, alpha, beta, st);
}

spmv_status_t launch_spmv32(spmv_matrix_t A, const float *x, float *y, cudaStream_t st) {
    if (A->variant == SPMV_VARIANT_SELL_WINDOW) return launch_window32(A, x, y, st);
    if (A->variant == SPMV_VARIANT_SELL_BULK) {
        bool launched = false;
        GB_TRY(launch_bulk32(A, x, y, st, &launched));
        if (launched) return SPMV_OK;
    }
    return launch_sell<float>(A, A->sell_val32.p, x, y, 1.0f, 0.0f, st);
}

spmv_status_t launch_spmv_csr64(spmv_matrix_t A, const double *x, double *y, cudaStream_t st) {
    if (A->n == 0) return SPMV_OK;
    spmv_csr<double><<<grid_for(A->n, 256), 256, 0, st>>>(A->n, A->row_ptr.p, A->col.p, A->val.p,
                                                          x, y);
    GB_LAUNCHED();
    return SPMV_OK;
}

spmv_status_t launch_permute(spmv_matrix_t A, int direction, int elem_bytes, const void *in,
                             void *out, cudaStream_t st) {
    if (A->n == 0) return SPMV_OK;
    const unsigned grid = grid_for(A->n, 256);
    if (!A->perm.p) {
        GB_CUDA(cudaMemcpyAsync(out, in, (size_t)A->n * elem_bytes, cudaMemcpyDeviceToDevice, st));
        return SPMV_OK;
    }
    if (elem_bytes == 8)
        permute_kernel<double><<<grid, 256, 0, st>>>(A->n, direction, A->perm.p,
                                                     (const double *)in, (double *)out);
    else
        permute_kernel<float><<<grid, 256, 0, st>>>(A->n, direction, A->perm.p,
                                                    (const float *)in, (float *)out);
    GB_LAUNCHED();
    return SPMV_OK;
}

spmv_status_t choose_variant(spmv_matrix_t A, cudaStream_t) {
    A->variant = A->opt.variant == SPMV_VARIANT_AUTO ? SPMV_VARIANT_SELL : A->opt.variant;
    A->window_words = A->variant == SPMV_VARIANT_SELL_WINDOW
                          ? window_capacity_words(A->has64() ? 8 : 4)
                          : 0;
    return SPMV_OK;
}

}  // namespace gb
