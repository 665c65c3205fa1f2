// convert.cu -- one-time pre-processing of a matrix on the device:
//   CSR validation; (reverse) Cuthill-McKee ordering by level-synchronous BFS (Sec. 4.1);
//   the symmetric permutation P A P^T; FP32 value copy; conversion to sliced ELLPACK with S
//   rows per slice, column-major inside a slice (Sec. 4.2); per-slice x range (Sec. 5.1).
// The paper applies these once per simulation, so their cost is amortised (Sec. 2, 4.1).
#include <cooperative_groups.h>

#include <climits>
#include <vector>

#include "common.cuh"

namespace cg = cooperative_groups;

namespace gb {
namespace {

constexpr int kT = 256;

inline unsigned blocks_for(int64_t n, int t = kT) {
    int64_t b = (n + t - 1) / t;
    return (unsigned)(b < 1 ? 1 : b);
}

// ---------------------------------------------------------------------------------------
// validation: row_ptr[0] = 0, row_ptr[n] = nnz, monotone, columns in range and strictly
// increasing inside each row.  Bits of *err: 1 ends, 2 monotone, 4 range, 8 order.
// ---------------------------------------------------------------------------------------
__global__ void validate_csr(int32_t n, int32_t n_cols, int64_t nnz, const int32_t *rp,
                             const int32_t *ci, int *err) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0 && (rp[0] != 0 || (int64_t)rp[n] != nnz)) atomicOr(err, 1);
    if (i >= n) return;
    int32_t a = rp[i], b = rp[i + 1];
    if (a > b || a < 0 || (int64_t)b > nnz) {
        atomicOr(err, 2);
        return;
    }
    int32_t prev = -1;
    for (int32_t k = a; k < b; ++k) {
        int32_t c = ci[k];
        if (c < 0 || c >= n_cols) {
            atomicOr(err, 4);
            return;
        }
        if (c <= prev) {
            atomicOr(err, 8);
            return;
        }
        prev = c;
    }
}

// ---------------------------------------------------------------------------------------
// Cuthill-McKee on the device.  A node's key is (degree, index).
// ---------------------------------------------------------------------------------------
__global__ void degree_kernel(int32_t n, const int32_t *rp, const int32_t *ci, int32_t *deg) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int32_t d = 0;
    for (int32_t k = rp[i]; k < rp[i + 1]; ++k) d += (ci[k] != (int32_t)i);
    deg[i] = d;
}

__device__ __forceinline__ unsigned long long node_key(const int32_t *deg, int32_t v) {
    return ((unsigned long long)(uint32_t)deg[v] << 32) | (uint32_t)v;
}

// a word that other CTAs write between barriers, from L2
__device__ __forceinline__ int32_t ld_l2(const int32_t *p) {
    int32_t v;
    asm volatile("ld.global.cg.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}

// *p = max(*p, x) if `on`: the value before, else x
__device__ __forceinline__ int32_t max_if(bool on, int32_t *p, int32_t x) {
    int32_t v = x;
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %3, 0;\n\t"
                 "@q atom.global.max.s32 %0, [%1], %2;\n\t}"
                 : "+r"(v) : "l"(p), "r"(x), "r"((int)on) : "memory");
    return v;
}
// *p += 1 if `on`, in the shared memory of any CTA of the cluster: the value before, else 0
__device__ __forceinline__ int32_t count_if(bool on, int *p) {
    int32_t v = 0;
    asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.s32 q, %2, 0;\n\t"
                 "@q atom.add.s32 %0, [%1], 1;\n\t}"
                 : "+r"(v) : "l"(p), "r"((int)on) : "memory");
    return v;
}

constexpr int kCmCluster = 16;
constexpr int kCmThreads = 1024;  // at most; see cm_order_device
constexpr int kCmPlaced = INT_MAX;  // stamp of a node that has its position
constexpr int kCmBatch = 6;     // row entries in flight per thread
constexpr int kCmComponents = 256;  // components that one launch orders
constexpr int kCmQueue = 4096;  // frontier nodes that a CTA keeps in shared memory
constexpr int kCmKids = 8;      // children of a node sorted in registers; more are sorted in memory
// Row entries per level, on average from the first one on, from which a component's levels go to
// the whole GPU.  A level costs a handful of launches and a read-back there (some 60 us), while the
// cluster's 16 SMs take some 0.2 ns per entry and level.  Whole set-up of connected random graphs, in
// ms, all levels launched from the host / all in the cluster / as here: 1M nodes of 7 entries 5.3 /
// 7.2 / 4.3, 4M 13.9 / 25.7 / 10.3, 300K of 43 14.6 / 21.1 / 8.7, 1M of 23 13.0 / 33.9 / 10.3.
constexpr int64_t kCmWide = 400000;

// How far an order has got.  A launch of cm_cluster ends early when it meets a component with wide
// levels: `wide` says whether while looking for its start node (from `start`) or between levels of
// its order, and then [ls, le) are the last level's positions.
enum { kCmNarrow, kCmWideSearch, kCmWideOrder };
struct CmProgress {
    int64_t placed, ls, le;
    int32_t bfs_id, spilled, wide, start;
};

// Smallest key that each CTA of the cluster found, in every CTA; two sets in turn, so that one can
// be written while another CTA still reads the last one.
struct CmKeys {
    unsigned long long key[2][kCmCluster];
    unsigned long long warp[kCmThreads / 32];
};

// A CTA's part of the frontier, one for the level that is read and one for the next, which the
// other CTAs write too.
struct CmFrontier {
    int32_t node[2][kCmQueue];
    // nodes that a BFS level has sent to this CTA: three words in turn, the next one cleared a level
    // ahead, when every CTA has passed the barrier after the last one read it
    int count[3];
    int full[3];  // whether a CTA's part was full, likewise
};

// What the CTAs of the cluster keep in step (every thread of every CTA holds the same values).
struct CmWalk {
    int32_t n;
    const int32_t *rp, *ci, *deg;
    int32_t *claim, *stamp, *queue, *perm;
    int32_t *spilled;  // BFS nodes in `queue`, those that found their CTA's frontier full
    int row, limit;    // mean row entries; nodes of a level of kCmWide of them
    CmKeys *keys;
    CmFrontier *front;
    cg::cluster_group cluster;
    int64_t gid, threads;  // threads are numbered across the CTAs: small levels use every SM
    int searches, levels;  // uses of the words above so far

    // up to kCmBatch neighbours of u from row entry k on, requested together (-1: none)
    __device__ __forceinline__ void load_row(int32_t u, int32_t k, int32_t end,
                                             int32_t (&v)[kCmBatch]) const {
#pragma unroll
        for (int j = 0; j < kCmBatch; ++j) v[j] = k + j < end ? ci[k + j] : -1;
#pragma unroll
        for (int j = 0; j < kCmBatch; ++j)
            if (v[j] == u) v[j] = -1;
    }

    __device__ __forceinline__ void take_min(unsigned long long &best, int32_t v) const {
        const unsigned long long k = node_key(deg, v);
        best = k < best ? k : best;
    }

    // smallest of the threads' keys
    __device__ __forceinline__ unsigned long long min_key(unsigned long long best) {
        const int w = searches++ & 1, ranks = (int)cluster.num_blocks();
        auto warp_min = [&] {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const unsigned long long k = __shfl_xor_sync(0xffffffffu, best, o);
                best = k < best ? k : best;
            }
        };
        warp_min();
        const int warps = blockDim.x >> 5;
        if ((threadIdx.x & 31) == 0) keys->warp[threadIdx.x >> 5] = best;
        __syncthreads();
        if (threadIdx.x < 32) {
            best = (int)threadIdx.x < warps ? keys->warp[threadIdx.x] : ~0ull;
            warp_min();
            if ((int)threadIdx.x < ranks)
                cluster.map_shared_rank(keys, threadIdx.x)->key[w][cluster.block_rank()] = best;
        }
        cluster.sync();
        for (int r = 0; r < ranks; ++r) best = keys->key[w][r] < best || r == 0 ? keys->key[w][r] : best;
        return best;
    }

    // Whether `levels_` levels of `nodes` nodes together, `last` of them in the last, are too wide for
    // the cluster (the average passes kCmWide at a level that does).
    __device__ __forceinline__ bool wide(int32_t last, int64_t nodes, int32_t levels_) const {
        return last > limit && nodes * row > kCmWide * levels_;
    }

    // BFS levels from r over nodes without a position: the number of levels, and the node of
    // the last one with the smallest key; false if they are too wide.  Ids grow, and a stamp only grows, so that one atomicMax
    // tells whether a node is new; it then goes to the CTA that its index hashes to.
    __device__ __forceinline__ bool bfs(int32_t r, int32_t id, int32_t *ecc, int32_t *pick) {
        const int ranks = (int)cluster.num_blocks(), lane = threadIdx.x & 31;
        const int shift = ranks == 16 ? 28 : 29;
        int mine = 0;  // nodes of the level in this CTA's frontier
        if (cluster.block_rank() == 0) {
            mine = 1;
            if (threadIdx.x == 0) {
                stamp[r] = id;
                front->node[levels & 1][0] = r;
            }
        }
        cluster.sync();
        int32_t ls = 0, le = 0;  // the level's nodes in `queue`
        int32_t depth = 0;
        auto owner = [&](int32_t v) {
            return cluster.map_shared_rank(front, (uint32_t)v * 2654435761u >> shift);
        };
        auto visit = [&](int32_t u, int w) {
            const int32_t b = rp[u + 1];
            for (int32_t k = rp[u]; k < b; k += kCmBatch) {
                int32_t v[kCmBatch], slot[kCmBatch];
                load_row(u, k, b, v);
                // (results are looked at after all of a kind have been requested: an atomic whose
                // result decides a branch waits for it, 1,000 clocks each)
                int32_t was[kCmBatch];
#pragma unroll
                for (int j = 0; j < kCmBatch; ++j) was[j] = max_if(v[j] >= 0, stamp + v[j], id);
#pragma unroll
                for (int j = 0; j < kCmBatch; ++j)
                    if (was[j] >= id) v[j] = -1;
#pragma unroll
                for (int j = 0; j < kCmBatch; ++j)
                    slot[j] = count_if(v[j] >= 0, &owner(v[j])->count[w]);
#pragma unroll
                for (int j = 0; j < kCmBatch; ++j) {
                    if (v[j] < 0) continue;
                    if (slot[j] < kCmQueue) {
                        owner(v[j])->node[~levels & 1][slot[j]] = v[j];
                    } else {
                        queue[atomicAdd(spilled, 1)] = v[j];
                        for (int r = 0; r < ranks; ++r)
                            cluster.map_shared_rank(front, r)->full[w] = 1;
                    }
                }
            }
        };
        int last = 0;  // the same of the level before
        int32_t last_ls = 0;
        int size = 0;      // nodes of the last level, and of all so far
        int64_t seen = 0;
        for (bool first = true;; first = false) {
            const int w = levels % 3;
            // how many nodes the level has is needed only once it has been visited
            const int sent = first ? lane == 0
                             : lane < ranks
                                 ? cluster.map_shared_rank(front, lane)->count[(levels + 2) % 3]
                                 : 0;
            const int share = mine + (le - ls + ranks - 1 - (int)cluster.block_rank()) / ranks;
            for (int i = threadIdx.x; i < share; i += blockDim.x)
                visit(i < mine ? front->node[levels & 1][i]
                               : ld_l2(queue + ls + (i - mine) * ranks + cluster.block_rank()),
                      w);
            if (threadIdx.x == 0) front->count[(levels + 1) % 3] = front->full[(levels + 1) % 3] = 0;
            cluster.sync();
            if (!__any_sync(0xffffffffu, sent > 0)) break;
            // (the level's size is looked at a level later, so that nothing waits for it)
            if (wide(size, seen, depth)) return false;
            size = __reduce_add_sync(0xffffffffu, sent);
            seen += size;
            last = mine;
            last_ls = ls;
            const int own = front->count[w];
            mine = own < kCmQueue ? own : kCmQueue;
            ls = le;
            if (front->full[w]) {
                const int all = lane < ranks ? cluster.map_shared_rank(front, lane)->count[w] : 0;
                le += __reduce_add_sync(0xffffffffu, all > kCmQueue ? all - kCmQueue : 0);
                const int next = __reduce_add_sync(0xffffffffu, all);
                if (wide(next, seen + next, depth + 1)) return false;
            }
            ++depth;
            ++levels;
        }
        // the level after the last one was empty
        unsigned long long best = ~0ull;
        for (int i = threadIdx.x; i < last; i += blockDim.x)
            take_min(best, front->node[~levels & 1][i]);
        for (int64_t i = last_ls + gid; i < ls; i += threads) take_min(best, ld_l2(queue + i));
        --depth;
        ++levels;
        if (gid == 0) *spilled = 0;
        *ecc = depth;
        *pick = (int32_t)(min_key(best) & 0xffffffffull);
        return true;
    }
};

// Children of frontier position p (the neighbours of its node u that no earlier position claimed):
// their number, and the first kCmKids keys, sorted.
__device__ __noinline__ int cm_kids(const CmWalk &w, int32_t p, int32_t u,
                                    unsigned long long (&key)[kCmKids]) {
#pragma unroll
    for (int j = 0; j < kCmKids; ++j) key[j] = ~0ull;
    int cnt = 0;
    const int32_t b = w.rp[u + 1];
    for (int32_t k = w.rp[u]; k < b; k += kCmBatch) {
        int32_t v[kCmBatch], c[kCmBatch], d[kCmBatch];
        w.load_row(u, k, b, v);
#pragma unroll
        for (int j = 0; j < kCmBatch; ++j) {
            c[j] = v[j] >= 0 ? ld_l2(w.claim + v[j]) : -1;
            d[j] = v[j] >= 0 ? w.deg[v[j]] : 0;
        }
#pragma unroll
        for (int i = 0; i < kCmBatch; ++i) {
            if (c[i] != p) continue;
            // insertion into the sorted list (a full list keeps the smallest)
            unsigned long long x = (unsigned long long)(uint32_t)d[i] << 32 | (uint32_t)v[i];
#pragma unroll
            for (int j = 0; j < kCmKids; ++j) {
                const unsigned long long lo = x < key[j] ? x : key[j];
                x = x < key[j] ? key[j] : x;
                key[j] = lo;
            }
            ++cnt;
        }
    }
    return cnt;
}

// The next level of the order: its first position, how many nodes each CTA takes, and where they
// are kept (in shared memory if every CTA's fit).
struct CmNext {
    int32_t first, run;
    int buf;
};
// Sets positions from `at` on, a few of them: position at + i is node i of `slot`.
struct CmSet {
    const CmWalk &w;
    const CmNext &next;
    int32_t at;
    int to, slot;
    __device__ __forceinline__ CmSet(const CmWalk &w_, const CmNext &next_, int32_t at_)
        : w(w_), next(next_), at(at_) {
        to = (at - next.first) / next.run;
        slot = at - next.first - to * next.run;
    }
    __device__ __forceinline__ void set(int i, int32_t v) const {
        w.perm[at + i] = v;
        w.stamp[v] = kCmPlaced;
        if (next.run > kCmQueue) return;
        int t = to, k = slot + i;
        while (k >= next.run) {
            k -= next.run;
            ++t;
        }
        w.cluster.map_shared_rank(w.front, t)->node[next.buf][k] = v;
    }
};

// The children of position p (its node u's neighbours that it claimed) to out, in increasing
// (degree, index): any number, sorted in place.  out is written by the calling thread alone.
// (Selecting them one by one, a row read per child: 2,000 hubs of 200 leaves in a chain 11.9 s
// with claims from L2, 6.1 s from L1; sorted 0.33 s.)
__device__ __noinline__ void cm_sort_kids(const int32_t *rp, const int32_t *ci, const int32_t *deg,
                                          const int32_t *claim, int32_t p, int32_t u, int32_t *out) {
    int cnt = 0;
    for (int32_t k = rp[u], b = rp[u + 1]; k < b; k += kCmBatch) {
        int32_t v[kCmBatch], c[kCmBatch];
#pragma unroll
        for (int j = 0; j < kCmBatch; ++j) v[j] = k + j < b ? ci[k + j] : u;
#pragma unroll
        for (int j = 0; j < kCmBatch; ++j) c[j] = v[j] != u ? ld_l2(claim + v[j]) : -1;
#pragma unroll
        for (int j = 0; j < kCmBatch; ++j)
            if (c[j] == p) out[cnt++] = v[j];
    }
    if (cnt <= 2 * kCmKids) {  // insertion
        for (int i = 1; i < cnt; ++i) {
            const int32_t x = out[i];
            const unsigned long long key = node_key(deg, x);
            int j = i;
            for (; j > 0 && node_key(deg, out[j - 1]) > key; --j) out[j] = out[j - 1];
            out[j] = x;
        }
        return;
    }
    // heap: the largest of out[0, end) goes to its end
    auto sift = [&](int at, int end) {
        const int32_t x = out[at];
        const unsigned long long key = node_key(deg, x);
        for (int kid; (kid = 2 * at + 1) < end; at = kid) {
            int32_t y = out[kid];
            unsigned long long ky = node_key(deg, y);
            if (kid + 1 < end) {
                const int32_t z = out[kid + 1];
                const unsigned long long kz = node_key(deg, z);
                if (kz > ky) {
                    y = z;
                    ky = kz;
                    ++kid;
                }
            }
            if (ky < key) break;
            out[at] = y;
        }
        out[at] = x;
    };
    for (int i = cnt / 2 - 1; i >= 0; --i) sift(i, cnt);
    for (int end = cnt - 1; end > 0; --end) {
        const int32_t x = out[end];
        out[end] = out[0];
        out[0] = x;
        sift(0, end);
    }
}

// Places the children of position p from position `at` on, in increasing (degree, index).
__device__ __forceinline__ void cm_place_kids(const CmWalk &w, const CmSet &set, int32_t p,
                                              int32_t u, int cnt,
                                              const unsigned long long (&key)[kCmKids]) {
    if (cnt <= kCmKids) {
#pragma unroll
        for (int j = 0; j < kCmKids; ++j)
            if (j < cnt) set.set(j, (int32_t)(key[j] & 0xffffffffull));
        return;
    }
    cm_sort_kids(w.rp, w.ci, w.deg, w.claim, p, u, w.perm + set.at);
    for (int t = 0; t < cnt; ++t) set.set(t, w.perm[set.at + t]);
}

// Cuthill-McKee from position io->placed on, up to max_components further components (so that a
// launch is short whatever the graph), in one thread-block cluster: the levels of a mesh are
// a few thousand nodes in some hundred steps, so what a level costs is its chain of dependent
// loads and its barriers.  A cluster barrier is a hardware one, and nothing returns to the host
// between levels.  The frontier lies in the CTAs' shared memory, spread over all of them, and is
// written there by whichever CTA finds a node; a search's step is then row bounds, row, one
// atomic per neighbour, a slot in the finder's choice of CTA and the barrier: 800 + 600 + 1,130 +
// 700 + 1,700 of its 6,600 clocks (3.3 us; 6 with the frontier in global memory, a look at each
// stamp before the atomic, and atomics that waited for one another).  A level of the order takes
// 5.9 us.  Whole set-up of 796K cells (1,038 levels of the start-node search, 353 of the order)
// 9.7 -> 6.4 ms, 48K 3.1 -> 2.2, 192K mixed 4.6 -> 3.7, 6M 40.6 -> 32.0.
template <int THREADS>
__global__ void __launch_bounds__(THREADS)
cm_cluster(int32_t n, const int32_t *rp, const int32_t *ci, const int32_t *deg, int32_t *claim,
           int32_t *stamp, int32_t *queue, int32_t *perm, int peripheral, int max_components,
           CmProgress *io) {
    __shared__ CmKeys keys;
    __shared__ CmFrontier front;
    __shared__ int totals[2][kCmCluster];
    __shared__ int warp_sums[THREADS / 32];
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = (int)cluster.block_rank(), ranks = (int)cluster.num_blocks();
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (threadIdx.x < 3) front.count[threadIdx.x] = front.full[threadIdx.x] = 0;
    CmWalk w{n, rp, ci, deg, claim, stamp, queue, perm, &io->spilled, rp[n] / n + 1,
             (int)(kCmWide / (rp[n] / n + 1)), &keys, &front,
             cluster,
             (int64_t)threadIdx.x * ranks + rank, (int64_t)ranks * THREADS, 0, 0};
    int32_t placed = (int32_t)io->placed;
    int32_t bfs_id = io->bfs_id;
    const int log_ranks = ranks == 16 ? 4 : 3;
    int turn = 0, wide = kCmNarrow;
    int32_t start = 0, ls = 0, le = 0;
    cluster.sync();
    if (w.gid == 0) io->spilled = 0;
    for (int comp = 0; comp < max_components && placed < n; ++comp) {
        // a node without a position is one that nothing has claimed
        unsigned long long best = ~0ull;
        for (int64_t i = w.gid; i < n; i += w.threads)
            if (ld_l2(claim + i) == INT_MAX) w.take_min(best, (int32_t)i);
        start = (int32_t)(w.min_key(best) & 0xffffffffull);
        if (peripheral) {
            const int32_t first = start;
            int32_t ecc = -1, pick = start;
            for (int searches = 0; searches <= 8; ++searches) {
                int32_t ecc2, pick2;
                if (!w.bfs(pick, bfs_id++, &ecc2, &pick2)) {
                    wide = kCmWideSearch;
                    start = first;
                    break;
                }
                if (ecc2 <= ecc) break;
                start = pick;
                ecc = ecc2;
                pick = pick2;
            }
            if (wide) break;
        }
        if (w.gid == 0) {
            claim[start] = -1;
            CmSet(w, CmNext{placed, 1, 0}, placed).set(0, start);
        }
        cluster.sync();
        ls = placed;
        le = placed + 1;
        int buf = 0;
        for (int32_t level = 1; le > ls; ++level) {
            // the CTAs take equal runs of the frontier, their threads `m` consecutive positions
            // each, so that the children's order is that of a scan over CTAs and threads
            const int32_t run = ((le - ls - 1) >> log_ranks) + 1;
            const int32_t m = (run + THREADS - 1) / THREADS;
            // counted from ls (positions up to n + kCmCluster THREADS would overflow)
            const int32_t size = le - ls, r1 = (rank + 1) * run < size ? (rank + 1) * run : size;
            const int32_t q0 = rank * run + (int)threadIdx.x * m;
            const int32_t p0 = ls + (q0 < r1 ? q0 : r1), p1 = ls + (q0 + m < r1 ? q0 + m : r1);
            const int32_t r0 = ls + rank * run;
            auto node = [&](int32_t p) {
                return run <= kCmQueue ? front.node[buf][p - r0] : ld_l2(perm + p);
            };
            // every neighbour of a frontier node records the earliest position; one that has its
            // own keeps the smaller claim of its parent
            int32_t u = -1, v[kCmBatch], d[kCmBatch];
            bool one = p1 - p0 == 1;  // one position, and a row that v holds
            for (int32_t p = p0; p < p1; ++p) {
                u = node(p);
                const int32_t b = rp[u + 1];
                for (int32_t k = rp[u]; k < b; k += kCmBatch) {
                    w.load_row(u, k, b, v);
#pragma unroll
                    for (int j = 0; j < kCmBatch; ++j)
                        if (v[j] >= 0) atomicMin(&claim[v[j]], p);
                    one = one && b - k <= kCmBatch;
                }
                one = one && rp[u] < b;
            }
            if (one) {
#pragma unroll
                for (int j = 0; j < kCmBatch; ++j) d[j] = v[j] >= 0 ? deg[v[j]] : 0;
            }
            cluster.sync();
            // children per thread, their scan over the cluster
            int mine = 0;
            unsigned long long key[kCmKids];
            if (one) {
                int32_t c[kCmBatch];
#pragma unroll
                for (int j = 0; j < kCmBatch; ++j) c[j] = v[j] >= 0 ? ld_l2(claim + v[j]) : -1;
#pragma unroll
                for (int j = 0; j < kCmBatch; ++j) {
                    if (c[j] != p0) v[j] = -1;
                    else ++mine;
                }
            } else {
                for (int32_t p = p0; p < p1; ++p) mine += cm_kids(w, p, node(p), key);
            }
            int incl = mine;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int x = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += x;
            }
            if (lane == 31) warp_sums[warp] = incl;
            __syncthreads();
            const int ws = lane < THREADS / 32 ? warp_sums[lane] : 0;
            int before = lane < warp ? ws : 0, all = ws;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                before += __shfl_xor_sync(0xffffffffu, before, o);
                all += __shfl_xor_sync(0xffffffffu, all, o);
            }
            turn ^= 1;
            if ((int)threadIdx.x < ranks)
                *cluster.map_shared_rank(&totals[turn][rank], threadIdx.x) = all;
            cluster.sync();
            int32_t at = le + before + incl - mine, total = 0;
            for (int r = 0; r < ranks; ++r) {
                const int x = totals[turn][r];
                if (r < rank) at += x;
                total += x;
            }
            const CmNext next{le, ((total - 1) >> log_ranks) + 1, buf ^ 1};
            if (one && mine) {
                const CmSet set(w, next, at);
                // a child's place: how many siblings have a smaller key
#pragma unroll
                for (int j = 0; j < kCmBatch; ++j) {
                    if (v[j] < 0) continue;
                    int rank_of = 0;
#pragma unroll
                    for (int i = 0; i < kCmBatch; ++i)
                        rank_of += v[i] >= 0 && (d[i] < d[j] || (d[i] == d[j] && v[i] < v[j]));
                    set.set(rank_of, v[j]);
                }
            } else if (mine) {
                for (int32_t p = p0; p < p1; ++p) {
                    const int32_t x = node(p);
                    const int cnt = p1 - p0 == 1 ? mine : cm_kids(w, p, x, key);
                    if (cnt) cm_place_kids(w, CmSet(w, next, at), p, x, cnt, key);
                    at += cnt;
                }
            }
            cluster.sync();
            buf ^= 1;
            ls = le;
            le += total;
            if (w.wide(total, le - placed, level + 1)) {
                wide = kCmWideOrder;
                break;
            }
        }
        placed = le;
        if (wide) break;
    }
    if (w.gid == 0) {
        io->placed = placed;
        io->bfs_id = bfs_id;
        io->wide = wide;
        io->start = start;
        io->ls = ls;
        io->le = le;
    }
    cluster.sync();  // no CTA leaves while another may use its shared memory
}

// ---- levels too wide for the cluster, a thread per node of the level; the same arrays ----------
__global__ void wide_seed(int32_t r, int32_t id, int32_t *stamp, int32_t *queue, int32_t *tail) {
    stamp[r] = id;
    queue[0] = r;
    *tail = 1;
}

// queue[ls, le): a BFS level; its unvisited neighbours without a position are appended
__global__ void wide_expand(const int32_t *rp, const int32_t *ci, int32_t id, int32_t *stamp,
                            int32_t *queue, int32_t ls, int32_t le, int32_t *tail) {
    const int64_t i = ls + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= le) return;
    const int32_t u = queue[i];
    for (int32_t k = rp[u]; k < rp[u + 1]; ++k) {
        const int32_t v = ci[k];
        if (v != u && stamp[v] < id && atomicMax(&stamp[v], id) < id) queue[atomicAdd(tail, 1)] = v;
    }
}

__global__ void wide_min_key(const int32_t *queue, int32_t ls, int32_t le, const int32_t *deg,
                             unsigned long long *out) {
    const int64_t i = ls + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < le) atomicMin(out, node_key(deg, queue[i]));
}

__global__ void wide_start(int32_t v, int32_t at, int32_t *claim, int32_t *stamp, int32_t *perm) {
    claim[v] = -1;
    stamp[v] = kCmPlaced;
    perm[at] = v;
}

__global__ void wide_claim(const int32_t *rp, const int32_t *ci, const int32_t *perm,
                           int32_t *claim, int32_t ls, int32_t le) {
    const int64_t p = ls + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= le) return;
    const int32_t u = perm[p];
    for (int32_t k = rp[u]; k < rp[u + 1]; ++k) {
        const int32_t v = ci[k];
        if (v != u && claim[v] > (int32_t)p) atomicMin(&claim[v], (int32_t)p);
    }
}

__global__ void wide_count(const int32_t *rp, const int32_t *ci, const int32_t *perm,
                           const int32_t *claim, int32_t ls, int32_t le, int64_t *counts) {
    const int64_t p = ls + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= le) return;
    const int32_t u = perm[p];
    int64_t c = 0;
    for (int32_t k = rp[u]; k < rp[u + 1]; ++k) c += ci[k] != u && claim[ci[k]] == (int32_t)p;
    counts[p - ls] = c;
}

__global__ void wide_place(const int32_t *rp, const int32_t *ci, const int32_t *deg,
                           const int32_t *claim, int32_t *stamp, int32_t *perm, int32_t ls,
                           int32_t le, const int64_t *offsets) {
    const int64_t p = ls + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= le) return;
    const int64_t first = offsets[p - ls];
    const int cnt = (int)(offsets[p - ls + 1] - first);
    if (!cnt) return;
    int32_t *out = perm + le + first;
    cm_sort_kids(rp, ci, deg, claim, (int32_t)p, perm[p], out);
    for (int t = 0; t < cnt; ++t) stamp[out[t]] = kCmPlaced;
}

__global__ void reverse_kernel(int32_t n, const int32_t *src, int32_t *dst) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) dst[i] = src[n - 1 - i];
}

__global__ void fill_i32(int32_t *p, int64_t n, int32_t v) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) p[i] = v;
}

// The arrays of an order: five of n words, then the progress.
struct CmArrays {
    int32_t n;
    const int32_t *rp, *ci;
    int32_t *deg, *claim, *stamp, *queue, *perm;
    CmProgress *progress;
};

// Component whose levels are too wide for cm_cluster, from where that left off (*g): its start node
// if need be, then its levels to the end.
spmv_status_t cm_wide_component(const CmArrays &a, bool peripheral, CmProgress *g,
                                cudaStream_t st) {
    struct Words {
        unsigned long long key;
        int32_t tail;
    } h, *d = nullptr;
    int64_t *counts = nullptr;
    auto read = [&]() -> spmv_status_t {
        GB_CUDA(cudaMemcpyAsync(&h, d, sizeof(Words), cudaMemcpyDeviceToHost, st));
        GB_CUDA(cudaStreamSynchronize(st));
        return SPMV_OK;
    };
    // levels from r: their number less one, and the node of the last one with the smallest key
    auto bfs = [&](int32_t r, int32_t *ecc, int32_t *pick) -> spmv_status_t {
        const int32_t id = g->bfs_id++;
        wide_seed<<<1, 1, 0, st>>>(r, id, a.stamp, a.queue, &d->tail);
        int32_t ls = 0, le = 1, last = 0;
        *ecc = -1;
        while (le > ls) {
            wide_expand<<<blocks_for(le - ls), kT, 0, st>>>(a.rp, a.ci, id, a.stamp, a.queue, ls,
                                                            le, &d->tail);
            GB_LAUNCHED();
            GB_TRY(read());
            last = ls;
            ls = le;
            le = h.tail;
            ++*ecc;
        }
        GB_CUDA(cudaMemsetAsync(&d->key, 0xff, sizeof(d->key), st));
        wide_min_key<<<blocks_for(ls - last), kT, 0, st>>>(a.queue, last, ls, a.deg, &d->key);
        GB_LAUNCHED();
        GB_TRY(read());
        *pick = (int32_t)(h.key & 0xffffffffull);
        return SPMV_OK;
    };
    spmv_status_t s = [&]() -> spmv_status_t {
        GB_CUDA(gb_malloc_async((void **)&d, sizeof(Words), st));
        GB_CUDA(gb_malloc_async((void **)&counts, sizeof(int64_t) * ((size_t)a.n + 1), st));
        if (g->wide == kCmWideSearch) {
            int32_t start = g->start;
            if (peripheral) {
                int32_t ecc = -1, pick = start;
                for (int searches = 0; searches <= 8; ++searches) {
                    int32_t ecc2, pick2;
                    GB_TRY(bfs(pick, &ecc2, &pick2));
                    if (ecc2 <= ecc) break;
                    start = pick;
                    ecc = ecc2;
                    pick = pick2;
                }
            }
            wide_start<<<1, 1, 0, st>>>(start, (int32_t)g->placed, a.claim, a.stamp, a.perm);
            GB_LAUNCHED();
            g->ls = g->placed;
            g->le = g->placed + 1;
        }
        int32_t ls = (int32_t)g->ls, le = (int32_t)g->le;
        while (le > ls) {
            const unsigned nb = blocks_for(le - ls);
            wide_claim<<<nb, kT, 0, st>>>(a.rp, a.ci, a.perm, a.claim, ls, le);
            wide_count<<<nb, kT, 0, st>>>(a.rp, a.ci, a.perm, a.claim, ls, le, counts);
            GB_LAUNCHED();
            GB_TRY(exclusive_scan_i64(counts, le - ls, st));
            wide_place<<<nb, kT, 0, st>>>(a.rp, a.ci, a.deg, a.claim, a.stamp, a.perm, ls, le,
                                          counts);
            GB_LAUNCHED();
            int64_t total = 0;
            GB_CUDA(cudaMemcpyAsync(&total, counts + (le - ls), sizeof(int64_t),
                                    cudaMemcpyDeviceToHost, st));
            GB_CUDA(cudaStreamSynchronize(st));
            ls = le;
            le += (int32_t)total;
        }
        g->placed = le;
        return SPMV_OK;
    }();
    if (d) cudaFreeAsync(d, st);
    if (counts) cudaFreeAsync(counts, st);
    return s;
}

spmv_status_t cm_order_device(int32_t n, const int32_t *rp, const int32_t *ci, bool reverse,
                              bool peripheral, int32_t *perm_out, cudaStream_t st) {
    if (n == 0) return SPMV_OK;
    int32_t *mem = nullptr;
    const size_t stride = ((size_t)n + 63) / 64 * 64;
    GB_CUDA(gb_malloc_async((void **)&mem, sizeof(int32_t) * 5 * stride + sizeof(CmProgress), st));
    const CmArrays a{n,          rp, ci, mem, mem + stride, mem + 2 * stride, mem + 3 * stride,
                     mem + 4 * stride, (CmProgress *)(mem + 5 * stride)};
    spmv_status_t s = [&]() -> spmv_status_t {
        const unsigned nb = blocks_for(n);
        degree_kernel<<<nb, kT, 0, st>>>(n, rp, ci, a.deg);
        fill_i32<<<nb, kT, 0, st>>>(a.claim, n, INT_MAX);
        fill_i32<<<nb, kT, 0, st>>>(a.stamp, n, -1);
        GB_LAUNCHED();
        GB_CUDA(cudaMemsetAsync(a.progress, 0, sizeof(CmProgress), st));
        // 512 threads per CTA leave registers for a row's loads in flight; the frontiers of
        // larger graphs (about 10K nodes from 1.5M on) keep 1,024 busy.  Whole set-up, ms, 512 /
        // 1,024: 48K cells 2.2 / 3.1, 796K 6.6 / 8.5, 3.1M 18.5 / 17.8, 6M 34.4 / 33.7.
        const bool large = n >= 1500000;
        auto *kern = large ? cm_cluster<1024> : cm_cluster<512>;
        GB_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1));
        cudaLaunchAttribute attr[1];
        attr[0].id = cudaLaunchAttributeClusterDimension;
        attr[0].val.clusterDim.x = kCmCluster;
        attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
        cudaLaunchConfig_t cfg{};
        cfg.gridDim = dim3(kCmCluster);
        cfg.blockDim = dim3(large ? 1024 : 512);
        cfg.stream = st;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
        int fits = 0;
        if (cudaOccupancyMaxActiveClusters(&fits, kern, &cfg) != cudaSuccess || fits < 1) {
            cudaGetLastError();
            attr[0].val.clusterDim.x = 8;  // the portable size
            cfg.gridDim = dim3(8);
        }
        CmProgress g{};
        while (g.placed < n) {
            GB_CUDA(cudaLaunchKernelEx(&cfg, kern, n, rp, ci, (const int32_t *)a.deg, a.claim,
                                       a.stamp, a.queue, a.perm, peripheral ? 1 : 0, kCmComponents,
                                       a.progress));
            GB_CUDA(cudaMemcpyAsync(&g, a.progress, sizeof(g), cudaMemcpyDeviceToHost, st));
            GB_CUDA(cudaStreamSynchronize(st));
            if (g.wide) {
                GB_TRY(cm_wide_component(a, peripheral, &g, st));
                GB_CUDA(cudaMemcpyAsync(a.progress, &g, sizeof(g), cudaMemcpyHostToDevice, st));
            }
        }
        if (reverse)
            reverse_kernel<<<nb, kT, 0, st>>>(n, a.perm, perm_out);
        else
            GB_CUDA(cudaMemcpyAsync(perm_out, a.perm, sizeof(int32_t) * n,
                                    cudaMemcpyDeviceToDevice, st));
        GB_LAUNCHED();
        return SPMV_OK;
    }();
    cudaFreeAsync(mem, st);
    return s;
}

// ---------------------------------------------------------------------------------------
// length sorting inside windows of sigma rows (sliced ELLPACK with a sorting scope, ref.
// MON10): rows taken in the order perm_in (nullptr = identity) are reordered inside each window
// by decreasing length, equal lengths keeping their order, so the slices of a window pad less.
// One CTA per window: bitonic sort of the unique keys (INT_MAX - length, position).
// ---------------------------------------------------------------------------------------
__global__ void sigma_sort_kernel(int32_t n, int32_t sigma, const int32_t *rp,
                                  const int32_t *perm_in, int32_t *perm_out) {
    extern __shared__ unsigned long long keys[];
    const int64_t w0 = (int64_t)blockIdx.x * sigma;
    const int cnt = (int)((n - w0) < sigma ? (n - w0) : sigma);
    for (int j = threadIdx.x; j < sigma; j += blockDim.x) {
        if (j < cnt) {
            const int32_t old = perm_in ? perm_in[w0 + j] : (int32_t)(w0 + j);
            const uint32_t len = (uint32_t)(rp[old + 1] - rp[old]);
            keys[j] = ((unsigned long long)(0x7fffffffu - len) << 32) | (uint32_t)j;
        } else {
            keys[j] = ~0ull;
        }
    }
    __syncthreads();
    for (int k = 2; k <= sigma; k <<= 1) {
        for (int jj = k >> 1; jj > 0; jj >>= 1) {
            for (int i = threadIdx.x; i < sigma; i += blockDim.x) {
                const int ixj = i ^ jj;
                if (ixj > i) {
                    const bool up = (i & k) == 0;
                    const unsigned long long a = keys[i], b = keys[ixj];
                    if ((a > b) == up) {
                        keys[i] = b;
                        keys[ixj] = a;
                    }
                }
            }
            __syncthreads();
        }
    }
    for (int j = threadIdx.x; j < cnt; j += blockDim.x) {
        const int32_t src = (int32_t)(keys[j] & 0xffffffffull);
        perm_out[w0 + j] = perm_in ? perm_in[w0 + src] : (int32_t)(w0 + src);
    }
}

// ---------------------------------------------------------------------------------------
// symmetric permutation B = P A P^T (perm[new] = old), rows sorted by new column
// ---------------------------------------------------------------------------------------
__global__ void inverse_perm(int32_t n, const int32_t *perm, int32_t *inv) {
    int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r < n) inv[perm[r]] = (int32_t)r;
}

__global__ void permuted_lengths(int32_t n, const int32_t *rp, const int32_t *perm,
                                 int64_t *len) {
    int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r < n) len[r] = rp[perm[r] + 1] - rp[perm[r]];
}

__global__ void i64_to_i32(const int64_t *a, int32_t *b, int64_t n) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) b[i] = (int32_t)a[i];
}

__global__ void permute_rows(int32_t n, const int32_t *rp, const int32_t *ci, const double *val,
                             const int32_t *perm, const int32_t *inv, const int32_t *rp_out,
                             int32_t *ci_out, double *val_out) {
    int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n) return;
    const int32_t old = perm[r];
    const int32_t a = rp[old];
    const int32_t len = rp[old + 1] - a;
    const int32_t base = rp_out[r];
    for (int32_t t = 0; t < len; ++t) {
        ci_out[base + t] = inv[ci[a + t]];
        val_out[base + t] = val[a + t];
    }
    for (int32_t t = 1; t < len; ++t) {  // insertion sort by column
        int32_t c = ci_out[base + t];
        double v = val_out[base + t];
        int32_t b = t - 1;
        while (b >= 0 && ci_out[base + b] > c) {
            ci_out[base + b + 1] = ci_out[base + b];
            val_out[base + b + 1] = val_out[base + b];
            --b;
        }
        ci_out[base + b + 1] = c;
        val_out[base + b + 1] = v;
    }
}

__global__ void to_f32(const double *a, float *b, int64_t n) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) b[i] = __double2float_rn(a[i]);
}

__global__ void bandwidth_kernel(int32_t n, const int32_t *rp, const int32_t *ci, int *out) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    int32_t a = rp[i], b = rp[i + 1];
    if (a == b) return;
    int32_t d0 = (int32_t)i - ci[a];
    int32_t d1 = ci[b - 1] - (int32_t)i;
    atomicMax(out, d0 > d1 ? d0 : d1);
}

// ---------------------------------------------------------------------------------------
// sliced ELLPACK (Sec. 4.2) and the per-slice x range (Sec. 5.1)
// ---------------------------------------------------------------------------------------
__global__ void slice_sizes(int32_t n, int32_t S, int32_t n_slices, const int32_t *rp,
                            int64_t *sp) {
    int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= n_slices) return;
    int32_t w = 0;
    int64_t r0 = s * S;
    for (int64_t r = r0; r < r0 + S && r < n; ++r) {
        int32_t len = rp[r + 1] - rp[r];
        w = len > w ? len : w;
    }
    sp[s] = (int64_t)S * w;
}

template <bool F64, bool F32>
__global__ void sell_scatter(int32_t n, int32_t S, int64_t n_pad, const int32_t *rp,
                             const int32_t *ci, const double *val, const float *val32,
                             const int64_t *sp, int32_t *scol, double *sval, float *sval32) {
    int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= n_pad) return;
    const int64_t s = r / S;
    const int64_t lane = r - s * S;
    const int64_t base = sp[s];
    const int64_t w = (sp[s + 1] - base) / S;
    const int32_t a = r < n ? rp[r] : 0;
    const int32_t len = r < n ? rp[r + 1] - a : 0;
    for (int64_t t = 0; t < w; ++t) {
        const int64_t at = base + t * S + lane;
        if (t < len) {
            scol[at] = ci[a + t];
            if (F64) sval[at] = val[a + t];
            if (F32) sval32[at] = val32[a + t];
        } else {
            scol[at] = -1;
            if (F64) sval[at] = 0.0;
            if (F32) sval32[at] = 0.0f;
        }
    }
}

__global__ void window_meta(int32_t n_slices, int32_t S, const int64_t *sp, const int32_t *scol,
                            int32_t *cs, int32_t *ce, int *max_span_width) {
    const int64_t s = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (s >= n_slices) return;
    int32_t lo = INT_MAX, hi = -1;
    for (int64_t at = sp[s] + lane; at < sp[s + 1]; at += 32) {
        int32_t c = scol[at];
        if (c < 0) continue;
        lo = c < lo ? c : lo;
        hi = c > hi ? c : hi;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        int32_t l2 = __shfl_xor_sync(0xffffffffu, lo, o);
        int32_t h2 = __shfl_xor_sync(0xffffffffu, hi, o);
        lo = l2 < lo ? l2 : lo;
        hi = h2 > hi ? h2 : hi;
    }
    if (lane == 0) {
        if (hi < 0) {
            cs[s] = 0;
            ce[s] = 0;
        } else {
            cs[s] = lo;
            ce[s] = hi + 1;
            atomicMax(max_span_width, hi + 1 - lo);
        }
        atomicMax(max_span_width + 1, (int)((sp[s + 1] - sp[s]) / S));
    }
}

// 16-bit columns relative to the slice's first column (Sec. 5.1); padding -> 0xFFFF
__global__ void relative_cols16(int32_t n_slices, const int64_t *sp, const int32_t *scol,
                                const int32_t *cs, uint16_t *out) {
    const int64_t s = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (s >= n_slices) return;
    const int32_t base = cs[s];
    for (int64_t at = sp[s] + lane; at < sp[s + 1]; at += 32) {
        const int32_t c = scol[at];
        out[at] = c < 0 ? (uint16_t)0xFFFFu : (uint16_t)(c - base);
    }
}

}  // namespace

spmv_status_t build_sell(spmv_matrix_t A, int S, cudaStream_t st) {
    NvtxRange nvtx("spmv_create/sliced_ellpack");
    const int32_t n = A->n;
    const int32_t n_slices = (int32_t)(((int64_t)n + S - 1) / S);
    size_t *tally = &A->bytes;
    A->S = S;
    A->n_slices = n_slices;
    GB_TRY(A->slice_ptr.alloc((size_t)n_slices + 1, tally));
    slice_sizes<<<blocks_for(n_slices), kT, 0, st>>>(n, S, n_slices, A->row_ptr.p, A->slice_ptr.p);
    GB_LAUNCHED();
    GB_TRY(exclusive_scan_i64(A->slice_ptr.p, n_slices, st));
    int64_t total = 0;
    GB_CUDA(cudaMemcpyAsync(&total, A->slice_ptr.p + n_slices, sizeof(int64_t),
                            cudaMemcpyDeviceToHost, st));
    GB_CUDA(cudaStreamSynchronize(st));
    A->sell_entries = total;
    A->mean_width = n_slices > 0 ? (float)((double)total / ((double)n_slices * S)) : 0.f;
    GB_TRY(A->sell_col.alloc((size_t)total, tally));
    if (A->has64()) GB_TRY(A->sell_val.alloc((size_t)total, tally));
    else A->sell_val.release(tally);
    if (A->has32()) GB_TRY(A->sell_val32.alloc((size_t)total, tally));
    else A->sell_val32.release(tally);
    const int64_t n_pad = (int64_t)n_slices * S;
    const unsigned nb = blocks_for(n_pad);
    if (A->has64() && A->has32())
        sell_scatter<true, true><<<nb, kT, 0, st>>>(n, S, n_pad, A->row_ptr.p, A->col.p, A->val.p,
                                                    A->val32.p, A->slice_ptr.p, A->sell_col.p,
                                                    A->sell_val.p, A->sell_val32.p);
    else if (A->has64())
        sell_scatter<true, false><<<nb, kT, 0, st>>>(n, S, n_pad, A->row_ptr.p, A->col.p, A->val.p,
                                                     nullptr, A->slice_ptr.p, A->sell_col.p,
                                                     A->sell_val.p, nullptr);
    else
        sell_scatter<false, true><<<nb, kT, 0, st>>>(n, S, n_pad, A->row_ptr.p, A->col.p, nullptr,
                                                     A->val32.p, A->slice_ptr.p, A->sell_col.p,
                                                     nullptr, A->sell_val32.p);
    GB_LAUNCHED();
    GB_TRY(A->col_start.alloc((size_t)n_slices, tally));
    GB_TRY(A->col_end.alloc((size_t)n_slices, tally));
    int *d_span = nullptr;  // max span, max width
    GB_CUDA(gb_malloc_async((void **)&d_span, 2 * sizeof(int), st));
    cudaMemsetAsync(d_span, 0, 2 * sizeof(int), st);
    window_meta<<<blocks_for((int64_t)n_slices * 32), kT, 0, st>>>(
        n_slices, S, A->slice_ptr.p, A->sell_col.p, A->col_start.p, A->col_end.p, d_span);
    spmv_status_t s = cuda_status(cudaGetLastError());
    int span_width[2] = {0, 0};
    if (s == SPMV_OK)
        s = cuda_status(cudaMemcpyAsync(span_width, d_span, 2 * sizeof(int),
                                        cudaMemcpyDeviceToHost, st));
    cudaFreeAsync(d_span, st);
    if (s == SPMV_OK) s = cuda_status(cudaStreamSynchronize(st));
    if (s != SPMV_OK) return s;
    const int span = span_width[0];
    A->max_span = span;
    A->max_width = span_width[1];
    GB_TRY(bulk_partition(A, st));
    if (!A->dev_status.p) {
        GB_TRY(A->dev_status.alloc(1, tally));
        GB_CUDA(cudaMemsetAsync(A->dev_status.p, 0, sizeof(int), st));
    }
    // 16-bit relative columns when every slice spans fewer than 65,535 columns
    const int want = A->opt.index_bits;
    A->sell_col16.release(tally);
    A->index_bits = 32;
    if (want != 32 && span < 65535 && total > 0) {
        GB_TRY(A->sell_col16.alloc((size_t)total, tally));
        relative_cols16<<<blocks_for((int64_t)n_slices * 32), kT, 0, st>>>(
            n_slices, A->slice_ptr.p, A->sell_col.p, A->col_start.p, A->sell_col16.p);
        GB_LAUNCHED();
        A->index_bits = 16;
    }
    // a product is a dependent launch that reads matrix entries before its dep_wait: its kernel
    // may start while a kernel that has not been waited for here still writes them
    GB_CUDA(cudaStreamSynchronize(st));
    return SPMV_OK;
}

spmv_status_t build_matrix(spmv_matrix_t A, const int32_t *d_rp, const int32_t *d_ci,
                           const double *d_val, cudaStream_t st) {
    const int32_t n = A->n;
    const int64_t nnz = A->nnz;
    size_t *tally = &A->bytes;

    // 1. validation
    {
        int *d_err = nullptr;
        GB_CUDA(gb_malloc_async((void **)&d_err, sizeof(int), st));
        cudaMemsetAsync(d_err, 0, sizeof(int), st);
        validate_csr<<<blocks_for(n), kT, 0, st>>>(n, A->n_cols, nnz, d_rp, d_ci, d_err);
        spmv_status_t s = cuda_status(cudaGetLastError());
        int err = 0;
        if (s == SPMV_OK)
            s = cuda_status(cudaMemcpyAsync(&err, d_err, sizeof(int), cudaMemcpyDeviceToHost, st));
        cudaFreeAsync(d_err, st);
        if (s == SPMV_OK) s = cuda_status(cudaStreamSynchronize(st));
        if (s != SPMV_OK) return s;
        if (err) return SPMV_ERR_INVALID_CSR;
    }

    GB_TRY(A->row_ptr.alloc((size_t)n + 1, tally));
    GB_TRY(A->col.alloc((size_t)nnz, tally));
    GB_TRY(A->val.alloc((size_t)nnz, tally));

    // 2. ordering (Sec. 4.1), optional length sorting inside windows, symmetric permutation
    NvtxRange nvtx_order("spmv_create/reorder");
    const bool reorder = A->opt.reorder != SPMV_REORDER_NONE;
    const int sigma = A->opt.sigma;
    if ((reorder || sigma > 0) && n > 0) {
        GB_TRY(A->perm.alloc((size_t)n, tally));
        if (reorder)
            GB_TRY(cm_order_device(n, d_rp, d_ci, A->opt.reorder == SPMV_REORDER_RCM,
                                   A->opt.peripheral != 0, A->perm.p, st));
        if (sigma > 0) {
            int32_t *tmp = nullptr;
            GB_CUDA(gb_malloc_async((void **)&tmp, sizeof(int32_t) * n, st));
            const unsigned windows = (unsigned)(((int64_t)n + sigma - 1) / sigma);
            sigma_sort_kernel<<<windows, 1024, sizeof(unsigned long long) * sigma, st>>>(
                n, sigma, d_rp, reorder ? A->perm.p : nullptr, tmp);
            spmv_status_t s = cuda_status(cudaGetLastError());
            if (s == SPMV_OK)
                s = cuda_status(cudaMemcpyAsync(A->perm.p, tmp, sizeof(int32_t) * n,
                                                cudaMemcpyDeviceToDevice, st));
            cudaFreeAsync(tmp, st);
            if (s != SPMV_OK) return s;
        }
        int32_t *inv = nullptr;
        int64_t *len = nullptr;
        GB_CUDA(gb_malloc_async((void **)&inv, sizeof(int32_t) * n, st));
        GB_CUDA(gb_malloc_async((void **)&len, sizeof(int64_t) * ((size_t)n + 1), st));
        const unsigned nb = blocks_for(n);
        inverse_perm<<<nb, kT, 0, st>>>(n, A->perm.p, inv);
        permuted_lengths<<<nb, kT, 0, st>>>(n, d_rp, A->perm.p, len);
        spmv_status_t s = cuda_status(cudaGetLastError());
        if (s == SPMV_OK) s = exclusive_scan_i64(len, n, st);
        if (s == SPMV_OK) {
            i64_to_i32<<<blocks_for((int64_t)n + 1), kT, 0, st>>>(len, A->row_ptr.p, (int64_t)n + 1);
            permute_rows<<<nb, kT, 0, st>>>(n, d_rp, d_ci, d_val, A->perm.p, inv, A->row_ptr.p,
                                            A->col.p, A->val.p);
            s = cuda_status(cudaGetLastError());
        }
        cudaFreeAsync(inv, st);
        cudaFreeAsync(len, st);
        if (s != SPMV_OK) return s;
    } else {
        GB_CUDA(cudaMemcpyAsync(A->row_ptr.p, d_rp, sizeof(int32_t) * ((size_t)n + 1),
                                cudaMemcpyDeviceToDevice, st));
        if (nnz) {
            GB_CUDA(cudaMemcpyAsync(A->col.p, d_ci, sizeof(int32_t) * nnz,
                                    cudaMemcpyDeviceToDevice, st));
            GB_CUDA(cudaMemcpyAsync(A->val.p, d_val, sizeof(double) * nnz,
                                    cudaMemcpyDeviceToDevice, st));
        }
    }

    // 3. FP32 copy of the values
    if (A->has32()) {
        GB_TRY(A->val32.alloc((size_t)nnz, tally));
        to_f32<<<blocks_for(nnz), kT, 0, st>>>(A->val.p, A->val32.p, nnz);
        GB_LAUNCHED();
    }

    // 4. bandwidth (reported; Sec. 4.1 defines it as the band width the reordering shrinks)
    {
        int *d_bw = nullptr;
        GB_CUDA(gb_malloc_async((void **)&d_bw, sizeof(int), st));
        cudaMemsetAsync(d_bw, 0, sizeof(int), st);
        bandwidth_kernel<<<blocks_for(n), kT, 0, st>>>(n, A->row_ptr.p, A->col.p, d_bw);
        spmv_status_t s = cuda_status(cudaGetLastError());
        int bw = 0;
        if (s == SPMV_OK)
            s = cuda_status(cudaMemcpyAsync(&bw, d_bw, sizeof(int), cudaMemcpyDeviceToHost, st));
        cudaFreeAsync(d_bw, st);
        if (s == SPMV_OK) s = cuda_status(cudaStreamSynchronize(st));
        if (s != SPMV_OK) return s;
        A->bandwidth = bw;
    }

    // 5. sliced ELLPACK + per-slice x range
    GB_TRY(build_sell(A, A->S, st));
    return SPMV_OK;
}

}  // namespace gb
