// S3 on the device: the lazy-greedy pivot selection of Algorithm 2 (Phase 2)
// computed in parallel rounds with the same result.
//
// The lazy greedy (max-heap on (gain, lower id), stale entries reinserted)
// selects, at every step, the uncovered vertex of largest key
// (|R_k(x) \ Covered|, -x).  Selecting y can change x's key or cover x only if
// y is in x's conflict set
//     Conf(x) = N_k(x) u R_k(x) u { N_k(z) : z in R_k(x), z uncovered }
// (y covers x iff x in R_k(y) iff y in N_k(x); y lowers x's gain iff y covers
// an uncovered z in R_k(x), i.e. y = z or y in N_k(z)), and the relation is
// symmetric.  A vertex whose key beats every uncovered member of its conflict
// set keeps its key until the sequential greedy reaches it, so the sequential
// greedy selects it with the same follower set F_x = R_k(x) \ Covered; such
// local maxima never conflict with each other, so one round selects all of
// them at once.  The global maximum is always a local maximum, so every round
// makes progress.
//
// A round by votes: every uncovered z votes for the vertex of largest key among
// itself and its uncovered N_k(z).  Conf(x) is the union of these sets over x
// itself and the uncovered z in R_k(x), so x beats its conflict set iff all of
// them vote for it: gain(x) + 1 votes (a vote weighs as often as N_k(z) names x,
// plus one for z = x, so repeated entries count as they do in the gain).  The
// gains are kept, not recomputed: covering y takes one from every vertex of
// N_k(y).  So a round gathers k words per uncovered vertex and touches R_k(x) of
// the selected x only; before, every uncovered x read its whole conflict set,
// |R_k(x)| * k keys by one thread, and hubs set the time of each round.
//
// The uncovered vertices are listed anew every round, and the last rounds, few
// vertices each, run in one launch of one thread-block cluster, which needs no host
// between rounds (all rounds of up to kTailMax vertices run there, of up to kSmallMax in
// one block; larger segments go on over the whole grid until that few are left, see
// launch_select_pivots).  What is left is the chain of dependent loads of each round, some
// 11 us.  S3 of 5,000 Gaussian rows 2.14 -> 0.41 ms, 2 x 500k SIFT-like rows 1.55 -> 0.71 ms, 300k
// DEEP-like rows in 5 segments 3.25 -> 1.90 ms.

#include <cooperative_groups.h>

#include "internal.h"

namespace rnsm {

namespace {

constexpr int32_t kCovered = -(1 << 30);   // gain of a covered vertex (and below)
constexpr int64_t kTailMax = 32768;
constexpr int kWide = 24;                  // reverse lists from here on take a warp
constexpr int kFullRounds = 16;            // rounds over the whole grid at a time
constexpr int64_t kNoLook = 98304;         // see launch_select_pivots
// 16 bytes of state each in one block's shared memory.  One block and the cluster, whole
// calls: 6,144 and 6,145 DEEP-like rows 226 and 238 us, Gaussian ones (36 rounds) 494 and 544;
// at 8,001 rows the cluster is ahead (318 against 348 us for S3 of a merge).
constexpr int64_t kSmallMax = 6144;
constexpr int kTailBlocks = 8, kTailThreads = 1024;

struct PivotState {
    int32_t *gain;    // |R_k(x) \ Covered|, or kCovered and below
    int32_t *votes;
    int32_t *snap;    // the gain at the start of the round
    int32_t *pivot_of;
    const int32_t *nplus;
    const int64_t *offs;
    const int32_t *ids;
    int32_t k_plus, k;
};

__global__ void piv_init_kernel(PivotState s, int64_t n, int32_t *list, PivotCtl *ctl) {
    for (int64_t x = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; x < n;
         x += (int64_t)gridDim.x * blockDim.x) {
        s.gain[x] = (int32_t)(s.offs[x + 1] - s.offs[x]);
        s.votes[x] = 0;
        s.pivot_of[x] = -2;
        list[x] = (int32_t)x;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        *ctl = PivotCtl();
        ctl->count[0] = (int32_t)n;
    }
}

// The state lies in global memory (read past L1: other blocks write it) or, for the
// one-block kernel, in shared memory with 16-bit lists.
template <bool kShared, class T>
__device__ __forceinline__ int32_t get(const T *p) {
    if constexpr (kShared) return (int32_t)*const_cast<const volatile T *>(p);
    else return __ldcg(p);
}
template <bool kShared, class T>
__device__ __forceinline__ void put(T *p, int32_t v) {
    if constexpr (kShared) *const_cast<volatile T *>(p) = (T)v;
    else __stcg(p, v);
}

// The vote of the uncovered z, of gain gz.
template <bool kShared>
__device__ __forceinline__ void vote(const PivotState &s, int32_t z, int32_t gz) {
    put<kShared>(s.snap + z, gz);
    int32_t best = z, gb = gz;
    int weight = 1;   // z's own
    const int32_t *nz = s.nplus + (int64_t)z * s.k_plus;
#pragma unroll 5
    for (int j = 0; j < s.k; ++j) {
        const int32_t y = __ldg(nz + j);
        if (y < 0) continue;
        const int32_t gy = get<kShared>(s.gain + y);
        if (y == best) ++weight;
        else if (gy > gb || (gy == gb && gy >= 0 && y < best)) {
            best = y;
            gb = gy;
            weight = 1;
        }
    }
    atomicAdd(s.votes + best, weight);
}

// Lists the uncovered vertices of cur[0..nc) in next and takes their votes;
// thread t of `threads` (whole warps).
template <bool kShared, class T>
__device__ __forceinline__ void vote_phase(const PivotState &s, const T *cur, int32_t nc, T *next, int32_t *n_next,
                                           int64_t t, int64_t threads) {
    const int lane = threadIdx.x & 31;
    for (int64_t i0 = t - lane; i0 < nc; i0 += threads) {
        const int64_t i = i0 + lane;
        const int32_t z = i < nc ? get<kShared>(cur + i) : -1;
        const int32_t gz = z >= 0 ? get<kShared>(s.gain + z) : kCovered;
        const bool open = gz >= 0;
        const unsigned m = __ballot_sync(0xffffffffu, open);
        int base = 0;
        if (lane == 0 && m) base = atomicAdd(n_next, __popc(m));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (!open) continue;
        put<kShared>(next + base + __popc(m & lanemask_lt()), z);
        vote<kShared>(s, z, gz);
    }
}

// Covers the selected x and its uncovered reverse neighbours, by G lanes; four entries
// a lane at a time, so that a long list is not a chain of one entry's loads after
// another's (entry lo - 1: x itself).
template <bool kShared, int G>
__device__ __forceinline__ void cover_list(const PivotState &s, int32_t x, int64_t lo, int64_t hi, int sub) {
    for (int64_t e0 = lo + sub - 1; e0 < hi; e0 += 4 * G) {
        int32_t y[4];
        bool todo[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int64_t e = e0 + q * G;
            y[q] = e >= hi ? -1 : e < lo ? x : __ldg(s.ids + e);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const bool self = q == 0 && e0 < lo;
            todo[q] = self || (y[q] >= 0 && y[q] != x && get<kShared>(s.gain + y[q]) >= 0);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q)   // (a vertex listed twice: once)
            if (todo[q]) todo[q] = atomicExch(s.gain + y[q], kCovered) >= 0;
#pragma unroll
        for (int q = 0; q < 4; ++q)
            if (todo[q]) __stcg(s.pivot_of + y[q], q == 0 && e0 < lo ? -1 : x);
        for (int c = 0; c < s.k; ++c) {
            int32_t w[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) w[q] = todo[q] ? __ldg(s.nplus + (int64_t)y[q] * s.k_plus + c) : -1;
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (w[q] >= 0) atomicSub(s.gain + w[q], 1);
        }
    }
}

__device__ __forceinline__ unsigned drop_lowest(unsigned m, int n) {
    for (int q = 0; q < n; ++q) m &= m - 1u;
    return m;
}

// Selects the vertices of next[0..n) that have all their votes: they become
// pivots, their uncovered reverse neighbours followers.  Eight lanes per
// selected vertex, a warp where the reverse list is long (a hub's list by eight
// lanes is a chain of |R_k| / 8 rounds of four dependent loads).
template <bool kShared, class T>
__device__ __forceinline__ void select_phase(const PivotState &s, const T *next, int32_t n, int64_t t, int64_t threads) {
    const int lane = threadIdx.x & 31, sub = lane & 7, grp = lane >> 3;
    for (int64_t i0 = t - lane; i0 < n; i0 += threads) {
        const int64_t i = i0 + lane;
        const int32_t x = i < n ? get<kShared>(next + i) : -1;
        bool sel = false;
        if (x >= 0) {
            sel = get<kShared>(s.votes + x) == get<kShared>(s.snap + x) + 1;
            put<kShared>(s.votes + x, 0);
        }
        int64_t lo = 0, hi = 0;
        if (sel) {
            lo = s.offs[x];
            hi = s.offs[x + 1];
        }
        const bool wide = sel && hi - lo >= kWide;
        unsigned m = __ballot_sync(0xffffffffu, sel && !wide);
        for (; m; m = drop_lowest(m, 4)) {
            const unsigned r = drop_lowest(m, grp);
            const int src = r ? __ffs(r) - 1 : lane;
            const int32_t xs = __shfl_sync(0xffffffffu, x, src);
            const int64_t l = __shfl_sync(0xffffffffu, lo, src), h = __shfl_sync(0xffffffffu, hi, src);
            if (r) cover_list<kShared, 8>(s, xs, l, h, sub);
            __syncwarp();
        }
        for (m = __ballot_sync(0xffffffffu, wide); m; m &= m - 1u) {
            const int src = __ffs(m) - 1;
            const int32_t xs = __shfl_sync(0xffffffffu, x, src);
            const int64_t l = __shfl_sync(0xffffffffu, lo, src), h = __shfl_sync(0xffffffffu, hi, src);
            cover_list<kShared, 32>(s, xs, l, h, lane);
            __syncwarp();
        }
    }
}

// The same over the whole grid.  A block appends its 256 entries at once: the list's order,
// which decides how far the rounds' accesses lie apart, breaks up eight times later than
// with an append a warp (4M DEEP-like rows 25.6 -> 15.2 ms, 500k SIFT-like ones 0.80 -> 0.70).
__global__ void __launch_bounds__(256) piv_vote_kernel(PivotState s, const int32_t *cur, int32_t *next, PivotCtl *ctl,
                                                       int round) {
    __shared__ int32_t count[8], base;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t nc = ctl->count[round];
    for (int64_t i0 = blockIdx.x * (int64_t)256; i0 < nc; i0 += (int64_t)gridDim.x * 256) {
        const int64_t i = i0 + threadIdx.x;
        const int32_t z = i < nc ? get<false>(cur + i) : -1;
        const int32_t gz = z >= 0 ? get<false>(s.gain + z) : kCovered;
        const bool open = gz >= 0;
        const unsigned m = __ballot_sync(0xffffffffu, open);
        if (lane == 0) count[warp] = __popc(m);
        __syncthreads();
        int before = 0, all = 0;
#pragma unroll
        for (int w = 0; w < 8; ++w) {
            before += w < warp ? count[w] : 0;
            all += count[w];
        }
        if (threadIdx.x == 0) base = all ? atomicAdd(&ctl->count[round + 1], all) : 0;
        __syncthreads();
        if (open) {
            put<false>(next + base + before + __popc(m & lanemask_lt()), z);
            vote<false>(s, z, gz);
        }
    }
}

__global__ void __launch_bounds__(256) piv_select_kernel(PivotState s, const int32_t *next, PivotCtl *ctl, int round) {
    const int32_t n = ctl->count[round + 1];
    if (n > 0 && blockIdx.x == 0 && threadIdx.x == 0) ++ctl->rounds;
    select_phase<false>(s, next, n, blockIdx.x * (int64_t)blockDim.x + threadIdx.x, (int64_t)gridDim.x * blockDim.x);
}

// The remaining rounds, by one cluster.  Each round has fewer uncovered vertices
// than the one before (else the lists are not those of one graph: error).
__global__ void __cluster_dims__(kTailBlocks, 1, 1) __launch_bounds__(kTailThreads)
    piv_tail_kernel(PivotState s, int32_t *cur, int32_t *next, PivotCtl *ctl, int round) {
    cooperative_groups::cluster_group cluster = cooperative_groups::this_cluster();
    const int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, threads = kTailBlocks * (int64_t)kTailThreads;
    int32_t nc = __ldcg(&ctl->count[round]), before = INT32_MAX, rounds = 0;
    int32_t *slot = &ctl->count[round];   // slot[1], slot[2], slot[3] take turns
    for (int r = 0;; ++r) {
        int32_t *n_next = slot + 1 + r % 3;
        vote_phase<false>(s, cur, nc, next, n_next, t, threads);
        cluster.sync();
        nc = __ldcg(n_next);
        if (nc == 0) break;
        if (nc >= before) {
            if (t == 0) ctl->stuck = 1;
            break;
        }
        before = nc;
        ++rounds;
        if (t == 0) __stcg(slot + 1 + (r + 2) % 3, 0);   // next but one: read by all a round ago
        select_phase<false>(s, next, nc, t, threads);
        cluster.sync();
        int32_t *sw = cur;
        cur = next;
        next = sw;
    }
    if (t == 0) ctl->rounds += rounds;
}

// All of it for up to kSmallMax vertices, by one block with the state in shared memory:
// a round's chain of dependent accesses then mostly costs tens of cycles instead of
// hundreds each (5,000 Gaussian rows, 32 rounds: 464 us by the cluster, now 340; 8,001
// DEEP-like rows: the cluster is faster by 30 us).
__global__ void __launch_bounds__(kTailThreads) piv_small_kernel(PivotState s, int32_t n, int32_t *pivots,
                                                                 int32_t *followers, PivotCtl *ctl) {
    extern __shared__ int32_t state[];
    __shared__ int32_t cnt[3], n_piv, n_fol;
    s.gain = state;
    s.votes = state + n;
    s.snap = state + 2 * n;
    uint16_t *cur = reinterpret_cast<uint16_t *>(state + 3 * n), *next = cur + n;
    const int t = threadIdx.x, lane = t & 31;
    for (int x = t; x < n; x += kTailThreads) {
        s.gain[x] = (int32_t)(s.offs[x + 1] - s.offs[x]);
        s.votes[x] = 0;
        cur[x] = (uint16_t)x;
    }
    if (t < 3) cnt[t] = 0;
    if (t == 0) n_piv = n_fol = 0;
    __syncthreads();
    int32_t nc = n, before = INT32_MAX, rounds = 0, stuck = 0;
    for (int r = 0;; ++r) {
        vote_phase<true>(s, cur, nc, next, &cnt[r % 3], t, kTailThreads);
        __syncthreads();
        nc = cnt[r % 3];
        if (nc == 0) break;
        if (nc >= before) {
            stuck = 1;
            break;
        }
        before = nc;
        ++rounds;
        if (t == 0) cnt[(r + 2) % 3] = 0;   // read by all a round ago
        select_phase<true>(s, next, nc, t, kTailThreads);
        __syncthreads();
        uint16_t *sw = cur;
        cur = next;
        next = sw;
    }
    __syncthreads();   // (pivot_of is this block's own writing)
    for (int x0 = t - lane; x0 < n; x0 += kTailThreads) {
        const int x = x0 + lane;
        const bool pv = x < n && s.pivot_of[x] == -1, fl = x < n && !pv;
        const unsigned mp = __ballot_sync(0xffffffffu, pv), mf = __ballot_sync(0xffffffffu, fl);
        int bp = 0, bf = 0;
        if (lane == 0) {
            bp = atomicAdd(&n_piv, __popc(mp));
            bf = atomicAdd(&n_fol, __popc(mf));
        }
        bp = __shfl_sync(0xffffffffu, bp, 0);
        bf = __shfl_sync(0xffffffffu, bf, 0);
        if (pv) pivots[bp + __popc(mp & lanemask_lt())] = x;
        if (fl) followers[bf + __popc(mf & lanemask_lt())] = x;
    }
    __syncthreads();
    if (t == 0) {
        *ctl = PivotCtl();
        ctl->n_pivots = (unsigned long long)n_piv;
        ctl->n_followers = (unsigned long long)n_fol;
        ctl->rounds = rounds;
        ctl->stuck = stuck;
    }
}

__global__ void piv_compact_kernel(int64_t n, const int32_t *pivot_of, int32_t *pivots, int32_t *followers,
                                   PivotCtl *ctl) {
    const int lane = threadIdx.x & 31;
    for (int64_t x0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x - lane; x0 < n;
         x0 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t x = x0 + lane;
        const bool pv = x < n && pivot_of[x] == -1, fl = x < n && !pv;
        const unsigned mp = __ballot_sync(0xffffffffu, pv), mf = __ballot_sync(0xffffffffu, fl);
        unsigned long long bp = 0, bf = 0;
        if (lane == 0) {
            if (mp) bp = atomicAdd(&ctl->n_pivots, (unsigned long long)__popc(mp));
            if (mf) bf = atomicAdd(&ctl->n_followers, (unsigned long long)__popc(mf));
        }
        bp = __shfl_sync(0xffffffffu, bp, 0);
        bf = __shfl_sync(0xffffffffu, bf, 0);
        if (pv) pivots[bp + __popc(mp & lanemask_lt())] = (int32_t)x;
        if (fl) followers[bf + __popc(mf & lanemask_lt())] = (int32_t)x;
    }
}

int grid_n(int64_t n) {
    int64_t g = (n + 255) / 256;
    if (g > 2048) g = 2048;
    return g < 1 ? 1 : (int)g;
}

}  // namespace

size_t pivot_tmp_bytes(int64_t n) { return 3 * (size_t)n * sizeof(int32_t); }

cudaError_t launch_select_pivots(const int32_t *nplus, int64_t n, int32_t k_plus, int32_t k, const int64_t *offs,
                                 const int32_t *ids, int32_t *pivot_of, int32_t *pivots, int32_t *followers,
                                 void *tmp, PivotCtl *ctl, cudaStream_t st) {
    PivotState s;
    s.gain = static_cast<int32_t *>(tmp);
    s.votes = s.gain + n;
    s.snap = s.votes + n;
    s.pivot_of = pivot_of;
    s.nplus = nplus;
    s.offs = offs;
    s.ids = ids;
    s.k_plus = k_plus;
    s.k = k;
    if (n <= kSmallMax) {
        const int smem = (int)(n * (3 * sizeof(int32_t) + 2 * sizeof(uint16_t)));
        const cudaError_t e = cudaFuncSetAttribute(piv_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                   (int)(kSmallMax * 16));
        if (e != cudaSuccess) return e;
        piv_small_kernel<<<1, kTailThreads, smem, st>>>(s, (int32_t)n, pivots, followers, ctl);
        note_launches(1);
        return cudaGetLastError();
    }
    // the output lists hold the uncovered vertices meanwhile
    int32_t *cur = pivots, *next = followers;
    const int g = grid_n(n);
    piv_init_kernel<<<g, 256, 0, st>>>(s, n, cur, ctl);
    // Rounds over the whole grid, sixteen at a time, until few enough are left for the
    // cluster's eight SMs: looked at (a wait, some 15 us) for segments over kNoLook.  Sixteen
    // rounds leave SIFT-like rows almost nothing at 500k, but most of 4M DEEP-like rows (52
    // rounds: 99.9 ms with the rest in the cluster, 15.2 now) and of Gaussian ones (500k, 124
    // rounds: 53.6 and 5.8 ms; 75k, not looked at: 3.6).
    int round = 0;
    int32_t left = (int32_t)n;
    while (n > kTailMax) {
        for (round = 0; round < kFullRounds; ++round) {
            piv_vote_kernel<<<g, 256, 0, st>>>(s, cur, next, ctl, round);
            piv_select_kernel<<<g, 256, 0, st>>>(s, next, ctl, round);
            int32_t *sw = cur;
            cur = next;
            next = sw;
        }
        note_launches(2 * round);
        if (n <= kNoLook) break;
        const int32_t before = left;
        cudaError_t e = cudaMemcpyAsync(&left, &ctl->count[round], sizeof(left), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) return e;
        if (left <= kTailMax || left >= before) break;   // (no progress: the cluster's kernel reports it)
        e = cudaMemcpyAsync(&ctl->count[0], &ctl->count[round], sizeof(left), cudaMemcpyDeviceToDevice, st);
        if (e == cudaSuccess) e = cudaMemsetAsync(&ctl->count[1], 0, sizeof(ctl->count) - sizeof(left), st);
        if (e != cudaSuccess) return e;
    }
    piv_tail_kernel<<<kTailBlocks, kTailThreads, 0, st>>>(s, cur, next, ctl, round);
    piv_compact_kernel<<<g, 256, 0, st>>>(n, pivot_of, pivots, followers, ctl);
    note_launches(3);
    return cudaGetLastError();
}

}  // namespace rnsm
