// Kernel templates and launchers of K1, the batched beam search; included by
// the translation units that instantiate them (with or without a job table, by
// code mode; compiled in parallel).
#pragma once
#include <float.h>

#include <algorithm>

#include "internal.h"

namespace rnsm {

namespace {

constexpr int kSearchWarps = 4;
constexpr int kBatch = 32;      // candidates evaluated per batch, one per lane

// Launch-shape variants (identical results): 0 = half the rows in flight and
// registers capped for 8 CTAs per SM (FP32 rows), 6 (filter) or 9 (exact codes, which
// have this shape only: 2 x 500k SIFT-like rows S1 4.13 ms; 8 CTAs 4.24, 10 with spills
// 4.41); 1 = the full rows in flight, 4 CTAs; 2 = a whole batch of rows in flight
// (as far as 128 registers hold it), 2 CTAs: for launches of so few queries that each
// warp's own chain of dependent loads decides their time.
// A tuned variant number v selects shape v & 1 and, if v & 2, the L2
// prefetch of the runner-up's neighbourhood during each expansion.
constexpr int kLatencyShape = 2;
template <int MODE, int VAR>
struct Variant {
    static constexpr int kMinBlocks = VAR == kLatencyShape ? 2
                                    : MODE == kCodeExact ? 9
                                    : MODE == kCodeFilter ? (VAR == 0 ? 6 : 4)
                                    : VAR == 0 ? 8 : 4;
};

template <int F4, int MODE, int VAR>
struct Layout {
    static constexpr int quarter = F4 / 4 > 0 ? F4 / 4 : 1;
    static constexpr int G = quarter >= 32 ? 32 : quarter >= 16 ? 16 : quarter >= 8 ? 8
                           : quarter >= 4 ? 4 : quarter >= 2 ? 2 : 1;
    static constexpr int V = (F4 + G - 1) / G;   // float4 per lane per row
    static constexpr int RPI = 32 / G;            // rows per step
    static constexpr int U0 = V <= 1 ? 8 : V <= 3 ? 4 : 2;   // steps in flight, shape 1
    static constexpr int UW = MODE == kCodeFilter ? (RPI >= 8 ? 1 : 2)   // few rows pass the codes
                            : VAR == 0 ? U0 / 2 : VAR == 1 ? U0 : 32 / V >= 8 ? 8 : 4;
    // a batch has 32 rows, so G steps cover it
    static constexpr int U = UW > G ? G : UW > 0 ? UW : 1;
    static_assert((U & (U - 1)) == 0 && U * RPI <= kBatch, "steps in flight");
};

// The same for code rows of 4 * F4 bytes: a lane takes 16 bytes of a row (24
// of the 768 as 16 + 8); the last 2 of a row of 96 bytes' 8 lanes take none.
template <int F4, int VAR>
struct CodeLayout {
    static constexpr int G = F4 <= 16 ? 4 : F4 <= 32 ? 8 : F4 <= 64 ? 16 : 32;
    static constexpr int W = F4 <= 128 ? 4 : 6;   // words per lane
    static constexpr int RPI = 32 / G;
    static constexpr int UW = VAR == kLatencyShape ? (F4 <= 128 ? 16 : 8) : F4 == 64 ? 8 : 4;
    static constexpr int U = UW > G ? G : UW;
    static_assert(W * G >= F4 && (W == 4 || F4 == W * G), "lanes cover a row");
};

// The visited table of a launch: 16-byte buckets, of ids (tag_shift 0) or of tags.
struct TableShape {
    uint32_t buckets;
    int32_t shift, tag_shift;
};

// ---- the visited table ---------------------------------------------------
// Ids in sets of two buckets of four (a bucket is one 16-byte shared load; -1
// empty, slots filled in order): an id's home bucket, then its sibling, and if
// both are full it replaces an entry of its home.  Forgetting an id costs its
// re-evaluation if the search meets it again, never a result: an evaluated
// vertex outside C is worse than the worst entry of C, and one inside C is
// found there before it is inserted (`lossy`).
__device__ __forceinline__ int4 lds4(const int32_t *p) {
    int4 v;
    asm volatile("ld.shared.v4.s32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
                 : "r"((uint32_t)__cvta_generic_to_shared(p))
                 : "memory");
    return v;
}

// Marks id (want lanes) and returns whether this lane is the one that has to
// evaluate it: the bucket is read first (most ids are there already), and a new
// one claims its slot by compare-and-swap, so an id listed twice goes to one lane.
__device__ __forceinline__ bool visit(int32_t *tab, uint32_t sets, int32_t id, bool want, bool &lossy) {
    const uint32_t h = (uint32_t)id * 0x9E3779B1u;
    const uint32_t home = 2u * __umulhi(h, sets) + ((h >> 7) & 1u);
    uint32_t bk = home;
    bool fresh = false, lost = false;
    // (a loop that the lanes leave together: with early exits it ran 3 times longer)
    while (__any_sync(0xffffffffu, want)) {
        if (want) {
            const int4 w = lds4(tab + 4 * bk);
            if (w.x == id || w.y == id || w.z == id || w.w == id) {
                want = false;
            } else if (w.w < 0) {
                const int32_t old = atomicCAS(&tab[4 * bk + (w.x >= 0) + (w.y >= 0) + (w.z >= 0)], -1, id);
                fresh = old == -1;
                want = !fresh && old != id;   // another id took the slot: look again
            } else if (bk == home) {
                bk ^= 1u;
            } else {
                tab[4 * home + ((h >> 9) & 3u)] = id;
                fresh = lost = true;
                want = false;
            }
        }
    }
    lossy = lossy || __any_sync(0xffffffffu, lost);
    return fresh;
}

// The same in half the memory, for beams over 64: a bucket of eight 16-bit tags is
// a set.  With ids below 2^b, x = id * odd mod 2^b is a bijection, and x * sets =
// set * 2^b + rest; within a set the rests are at least `sets` apart, so rest >>
// log2(sets) tells its ids apart: as long as it has 15 bits (all ones is empty), tag and
// set are the id.  shift = 32 - b; tag_shift = shift + log2(sets), rounded down.
__device__ __forceinline__ bool visit_tags(int32_t *tab, uint32_t sets, int shift, int tag_shift, int32_t id, bool want,
                                           bool &lossy) {
    constexpr uint32_t kHigh = 0x80008000u;
    const uint32_t x = ((uint32_t)id * 0x9E3779B1u) << shift;
    const uint32_t set = __umulhi(x, sets), tag = (x * sets) >> tag_shift, both = tag * 0x10001u;
    auto zero_half = [](uint32_t v) { return (v - 0x00010001u) & ~v & kHigh; };   // non-zero iff a half of v is zero
    unsigned short *slots = reinterpret_cast<unsigned short *>(tab + 4 * set);
    bool fresh = false, lost = false;
    while (__any_sync(0xffffffffu, want)) {
        if (want) {
            const int4 w = lds4(tab + 4 * set);
            const uint32_t a = (uint32_t)w.x, b = (uint32_t)w.y, c = (uint32_t)w.z, d = (uint32_t)w.w;
            const int room = __popc((a & kHigh) >> 15 | (b & kHigh) >> 14 | (c & kHigh) >> 13 | (d & kHigh) >> 12);
            if (zero_half(a ^ both) | zero_half(b ^ both) | zero_half(c ^ both) | zero_half(d ^ both)) {
                want = false;
            } else if (room > 0) {
                const unsigned short old = atomicCAS(slots + 8 - room, (unsigned short)0xffffu, (unsigned short)tag);
                fresh = old == 0xffffu;
                want = !fresh && old != tag;   // another id took the slot: look again
            } else {
                slots[(x >> 9) & 7u] = (unsigned short)tag;
                fresh = lost = true;
                want = false;
            }
        }
    }
    lossy = lossy || __any_sync(0xffffffffu, lost);
    return fresh;
}

// ---- the candidate set C ---------------------------------------------------
// Sorted ascending, one 64-bit key per entry, entry i in register i / 32 of
// lane i % 32: (order-preserving bits of the distance) << 32 | id << 1 |
// expanded.  Empty entries are all ones (and count as expanded).  The array
// holds 32 * PER >= ef entries; those from rank ef on are leftovers that no
// longer take part (ranks only grow).
typedef unsigned long long beam_t;

__device__ __forceinline__ uint32_t order_bits(float d) {
    const uint32_t b = __float_as_uint(d);
    return b ^ ((uint32_t)((int32_t)b >> 31) | 0x80000000u);
}
__device__ __forceinline__ float unorder_bits(uint32_t u) {
    return __uint_as_float((u & 0x80000000u) ? u ^ 0x80000000u : ~u);
}

// In a sorted array the insertion of K is new[i] = min(old[i], max(old[i - 1], K)).
template <int PER>
__device__ __forceinline__ void beam_insert(beam_t (&k)[PER], beam_t K, bool lossy) {
    const int lane = threadIdx.x & 31;
    if (lossy) {   // K may be in C already, expanded or not
        bool dup = false;
#pragma unroll
        for (int t = 0; t < PER; ++t) dup = dup || (k[t] ^ K) <= 1ull;
        if (__any_sync(0xffffffffu, dup)) return;
    }
    beam_t before = 0ull;   // the last entry of the register before
#pragma unroll
    for (int t = 0; t < PER; ++t) {
        // (with several registers, those whose entries all precede K stay as they are)
        if (PER > 2 && __all_sync(0xffffffffu, k[t] < K)) continue;
        beam_t prev = __shfl_sync(0xffffffffu, k[t], (lane + 31) & 31);
        const beam_t last = prev;
        if (lane == 0) prev = before;
        before = last;
        const beam_t up = prev > K ? prev : K;
        k[t] = k[t] < up ? k[t] : up;
    }
}

// Entry i of C (uniform i), in every lane.
template <int PER>
__device__ __forceinline__ beam_t beam_at(const beam_t (&k)[PER], int i) {
    beam_t v = k[0];
#pragma unroll
    for (int t = 1; t < PER; ++t)
        if (i >= 32 * t) v = k[t];
    return __shfl_sync(0xffffffffu, v, i & 31);
}

// Keys of up to 32 candidates (one per lane, all ones none) into C.  Few go in
// one by one (a chain of about 90 cycles each); from kMany on all at once by
// their ranks, through the warp's scratch of 32 * PER keys: entry i moves up by
// the number of new keys below it, a new key goes behind the entries and the new
// keys below it.
constexpr int kMany = 4;
template <int PER>
__device__ __forceinline__ void beam_add(beam_t (&k)[PER], beam_t K, beam_t &worst, int ef, bool lossy,
                                         beam_t *scratch) {
    unsigned s = __ballot_sync(0xffffffffu, K < worst);
    if (s == 0u) return;
    const int lane = threadIdx.x & 31;
    if (lossy || __popc(s) < kMany) {
        do {
            const int src = __ffs(s) - 1;
            s &= s - 1u;
            beam_insert<PER>(k, __shfl_sync(0xffffffffu, K, src), lossy);
        } while (s);
    } else {
        const bool in = (s >> lane) & 1u;
        int up[PER], at = 0;
#pragma unroll
        for (int t = 0; t < PER; ++t) up[t] = 0;
        do {
            const int src = __ffs(s) - 1;
            s &= s - 1u;
            const beam_t N = __shfl_sync(0xffffffffu, K, src);
            int below = 0;
#pragma unroll
            for (int t = 0; t < PER; ++t) {
                const bool lt = k[t] < N;
                up[t] += lt ? 0 : 1;
                below += __popc(__ballot_sync(0xffffffffu, lt));
            }
            at += lane == src ? below : N < K ? 1 : 0;
        } while (s);
#pragma unroll
        for (int t = 0; t < PER; ++t)
            if (lane + 32 * t + up[t] < 32 * PER) scratch[lane + 32 * t + up[t]] = k[t];
        if (in && at < 32 * PER) scratch[at] = K;
        __syncwarp();
#pragma unroll
        for (int t = 0; t < PER; ++t) k[t] = scratch[lane + 32 * t];
        __syncwarp();
    }
    worst = beam_at<PER>(k, ef - 1);
}

// This lane's words of a code row.
template <int F4, int VAR>
__device__ __forceinline__ void code_words(const uint8_t *row, int sub, uint32_t (&x)[CodeLayout<F4, VAR>::W]) {
    constexpr int G = CodeLayout<F4, VAR>::G, W = CodeLayout<F4, VAR>::W;
    if (F4 < 4 * G && sub >= F4 / 4) sub = 0;   // idle lanes of a 96-byte row: any word
    const uint4 v = __ldg(reinterpret_cast<const uint4 *>(row) + sub);
    x[0] = v.x;
    x[1] = v.y;
    x[2] = v.z;
    x[3] = v.w;
    if (W == 6) {
        const uint2 t = __ldg(reinterpret_cast<const uint2 *>(row + 16 * G) + sub);
        x[W - 2] = t.x;
        x[W - 1] = t.y;
    }
}

// Adds the group's partial sums v[u] of its U rows in the tree of lane
// distances G/2, ..., 1.  Every step hands half of the rows to each half of the
// group, so the same sums take U - 1 + log2(G / U) exchanges instead of
// U * log2(G).  The lane ends with the sum of row `mine` in v[0]; `lead`: it is
// the first of the lanes that hold it.
template <int G, int U, class T>
__device__ __forceinline__ void group_sums(T (&v)[U], int sub, int &mine, bool &lead) {
    mine = 0;
    lead = true;
#pragma unroll
    for (int off = G / 2, left = U; off > 0; off >>= 1) {
        const bool hi = (sub & off) != 0;
        if (left > 1) {
            left >>= 1;
#pragma unroll
            for (int u = 0; u < left; ++u) {
                const T give = hi ? v[u] : v[u + left];
                const T keep = hi ? v[u + left] : v[u];
                v[u] = keep + __shfl_xor_sync(0xffffffffu, give, off);
            }
            mine += hi ? left : 0;
        } else {
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], off);
            lead = lead && !hi;
        }
    }
}

// The query's FP32 row: this lane's float4 in registers, or, where few rows need
// it, the whole row in the warp's shared memory.
template <int F4, int MODE, int VAR>
struct QueryRow {
    using Lay = Layout<F4, MODE, VAR>;
    static constexpr bool kShared = MODE == kCodeFilter;
    static constexpr int kRegs = MODE == kCodeNone ? Lay::V : 1;
    float4 r[kRegs];
    const float4 *s;
    __device__ __forceinline__ float4 at(int j, int sub) const { return kShared ? s[sub + Lay::G * j] : r[kShared ? 0 : j]; }
};

// The FP32 distances of rows ids[0..c) to the query, and those that beat the
// worst entry of a full C (empty entries are beaten by everything) into C.
// Each lane of a group of G sums its share of a row's dimensions in order, the
// group adds them in a tree: one order of additions, whatever the shape.
template <int F4, int PER, int MODE, int VAR>
__device__ __forceinline__ void eval_rows(const SearchArgs &a, const float *base, const int32_t *ids, int c,
                                          const QueryRow<F4, MODE, VAR> &q, beam_t (&k)[PER],
                                          beam_t &worst, bool lossy, beam_t *scratch) {
    using Lay = Layout<F4, MODE, VAR>;
    constexpr int G = Lay::G, V = Lay::V, RPI = Lay::RPI, U = Lay::U;
    const int lane = threadIdx.x & 31;
    const int grp = lane / G, sub = lane % G;
    for (int b0 = 0; b0 < c; b0 += RPI * U) {
        // rows past the last one repeat it (the same addresses: no traffic)
        float4 x[U][V];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (u > 0 && b0 + u * RPI >= c) continue;   // uniform: x[u] is not looked at
            const float *row = base + (int64_t)ids[min(b0 + u * RPI + grp, c - 1)] * (4 * F4) + 4 * sub;
#pragma unroll
            for (int j = 0; j < V; ++j)
                if (G * (j + 1) <= F4 || sub + G * j < F4) x[u][j] = ldg4(row + 4 * G * j);
        }
        float acc[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            acc[u] = 0.f;
            if (a.metric == 0) {
#pragma unroll
                for (int j = 0; j < V; ++j)
                    if (G * (j + 1) <= F4 || sub + G * j < F4) acc[u] = l2_acc(acc[u], q.at(j, sub), x[u][j]);
            } else {
#pragma unroll
                for (int j = 0; j < V; ++j)
                    if (G * (j + 1) <= F4 || sub + G * j < F4) acc[u] = ip_acc(acc[u], q.at(j, sub), x[u][j]);
            }
        }
        int mine;
        bool lead;
        group_sums<G, U>(acc, sub, mine, lead);
        const int r = b0 + mine * RPI + grp;
        beam_t K = ~0ull;
        if (lead && r < c) {
            const float d = a.metric == 0 ? acc[0] : 1.0f - acc[0];
            K = ((beam_t)order_bits(d) << 32) | ((uint32_t)ids[r] << 1);
        }
        beam_add<PER>(k, K, worst, a.ef, lossy, scratch);
    }
}

// The code distances S of rows ids[0..c).  kCodeExact: they are the distances
// and go into C.  kCodeFilter: ids whose S is at most `limit` are written to
// `pass`; returns their number.
template <int F4, int PER, int MODE, int VAR>
__device__ __forceinline__ int eval_codes(const SearchArgs &a, const uint8_t *codes, const int32_t *ids, int c,
                                          const uint32_t (&q)[CodeLayout<F4, VAR>::W], int32_t qq, float limit,
                                          int32_t *pass, beam_t (&k)[PER], beam_t &worst, bool lossy,
                                          beam_t *scratch) {
    using Lay = CodeLayout<F4, VAR>;
    constexpr int G = Lay::G, W = Lay::W, RPI = Lay::RPI, U = Lay::U;
    const int lane = threadIdx.x & 31;
    const int grp = lane / G, sub = lane % G;
    int np = 0;
    for (int b0 = 0; b0 < c; b0 += RPI * U) {
        uint32_t x[U][W];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            if (u > 0 && b0 + u * RPI >= c) continue;   // uniform: x[u] is not looked at
            const uint8_t *row = codes + (int64_t)ids[min(b0 + u * RPI + grp, c - 1)] * (4 * F4);
            code_words<F4, VAR>(row, sub, x[u]);
        }
        // S = q.q + x.x - 2 q.x, in integers
        int32_t S[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
            uint32_t xx = 0u, xq = 0u;
#pragma unroll
            for (int j = 0; j < W; ++j) {
                xx = __dp4a(x[u][j], x[u][j], xx);
                xq = __dp4a(x[u][j], q[j], xq);
            }
            S[u] = qq + (int32_t)xx - 2 * (int32_t)xq;
            if (F4 < W * G && sub >= F4 / W) S[u] = 0;
        }
        int mine;
        bool lead;
        group_sums<G, U>(S, sub, mine, lead);
        const int r = b0 + mine * RPI + grp;
        const bool live = lead && r < c;
        const float d = (float)S[0];
        if (MODE == kCodeExact) {
            beam_t K = ~0ull;
            if (live) K = ((beam_t)order_bits(d) << 32) | ((uint32_t)ids[r] << 1);
            beam_add<PER>(k, K, worst, a.ef, lossy, scratch);
        } else {
            const bool ok = live && !(d > limit);
            const unsigned m = __ballot_sync(0xffffffffu, ok);
            if (ok) pass[np + __popc(m & lanemask_lt())] = ids[r];
            np += __popc(m);
        }
    }
    return np;
}

// The code distance from which a row is known not to beat `worst`: the row's
// FP32 distance exceeds w when its distance proper exceeds w by the roundings of
// the FP32 sum (under 5e-5 of the sum's terms at 768 dimensions, taken as 1e-4).
// L2: s * sqrt(S) - err > sqrt(w (1 + 1e-4)).  Inner product: 1 - <x, q> =
// (||x - q||^2 + 2 - ||x||^2 - ||q||^2) / 2, the norms at most norm2.
__device__ __forceinline__ float code_limit(const CodeParams &cp, int metric, beam_t worst) {
    if (worst == ~0ull) return INFINITY;
    const float w = unorder_bits((uint32_t)(worst >> 32));
    const float d2 = metric == 0 ? w * 1.0001f : 2.f * (w + 1e-4f * cp.norm2 + 1e-6f) - 2.f + 2.f * cp.norm2;
    const float t = (sqrtf(fmaxf(d2, 0.f)) + cp.err) * cp.inv_scale;
    return t * t * 1.0001f + 1.f;
}

// JOBS: query g of the launch belongs to the job j with
// jobs[j].q_begin <= g < jobs[j + 1].q_begin and is query g - q_begin of that
// job; the job's fields replace the launch's (one launch, many pairs).  They
// are read from the warp's shared copy of the job where they are needed: held
// in registers across a query they cost 40 of them.
template <class T>
__device__ __forceinline__ T fresh_read(const T &v) { return *const_cast<const volatile T *>(&v); }
#define JF(f) (JOBS ? fresh_read(J->f) : a.f)

// Shared memory: per warp the visited table (16 bytes a bucket), then the batch's
// new ids and those that pass the codes, scratch for C (and, for the ids that
// pass, the query's row).
__host__ __device__ constexpr size_t warp_smem_bytes(uint32_t buckets, int efmax, int row_float4) {
    return ((size_t)buckets * 4 + 2 * kBatch) * sizeof(int32_t) + (size_t)efmax * sizeof(beam_t) +
           (size_t)row_float4 * sizeof(float4);
}

template <int F4, int EFMAX, int MODE, int VAR, bool JOBS>
__global__ void __launch_bounds__(kSearchWarps * 32, Variant<MODE, VAR>::kMinBlocks)
search_kernel(const SearchArgs a, const TableShape table, int prefetch) {
    using Lay = Layout<F4, MODE, VAR>;
    using CLay = CodeLayout<F4, VAR>;
    constexpr int G = Lay::G, PER = EFMAX / 32;
    extern __shared__ __align__(16) unsigned char smem[];
    const int lane = threadIdx.x & 31;
    const int warp = threadIdx.x >> 5;
    if (a.gate && (*a.gate & 3)) return;   // the inputs did not pass their checks
    int32_t *tab = reinterpret_cast<int32_t *>(smem + (size_t)warp * warp_smem_bytes(table.buckets, EFMAX, MODE == kCodeFilter ? F4 : 0));
    int32_t *ci = tab + table.buckets * 4;
    int32_t *pass = ci + kBatch;
    beam_t *scratch = reinterpret_cast<beam_t *>(pass + kBatch);
    float4 *qrow_s = reinterpret_cast<float4 *>(scratch + EFMAX);
    const int sub = lane % G;
    CodeParams cp;
    if (MODE == kCodeFilter) cp = *a.code_params;
    __shared__ SearchJob sjob[JOBS ? kSearchWarps : 1];

    unsigned long long ndc_total = 0, nexp_total = 0;
    int claim = 0;
    if (lane == 0) claim = atomicAdd(a.work, 1);
    for (;;) {
        const int qi = __shfl_sync(0xffffffffu, claim, 0);
        if (qi >= a.nq) break;
        // the next query: claimed now, while others have work enough, so that the
        // claim's latency is this search; towards the end only when it is done
        const bool early = (int64_t)qi + (int64_t)gridDim.x * kSearchWarps < a.nq;
        if (early && lane == 0) claim = atomicAdd(a.work, 1);
        int64_t gi = a.q0 + qi;  // index in the whole batch (JOBS: in its job)
        const SearchJob *J = nullptr;
        if (JOBS) {
            int lo = 0, hi = a.n_jobs - 1;
            while (lo < hi) {
                const int mid = (lo + hi + 1) >> 1;
                if (a.jobs[mid].q_begin <= gi) lo = mid; else hi = mid - 1;
            }
            // the job's fields go to this warp's shared slot and are read from
            // there when needed (no registers held across the query)
            static_assert(sizeof(SearchJob) % 4 == 0 && sizeof(SearchJob) <= 128, "job copy");
            const int32_t *src = reinterpret_cast<const int32_t *>(a.jobs + lo);
            int32_t *dst = reinterpret_cast<int32_t *>(&sjob[warp]);
            if (lane < (int)(sizeof(SearchJob) / 4)) dst[lane] = src[lane];
            __syncwarp();
            J = &sjob[warp];
            gi -= J->q_begin;
        }
        const int32_t *qidx = JF(qidx);
        const int32_t qrow = qidx ? qidx[gi] : (int32_t)gi;

        QueryRow<F4, MODE, VAR> q;
        if (MODE != kCodeExact) {
            const float *qv = JF(qvecs) + (int64_t)qrow * (4 * F4);
            if (q.kShared) {
                for (int f = lane; f < F4; f += 32) qrow_s[f] = ldg4(qv + 4 * f);
                q.s = qrow_s;
            } else {
#pragma unroll
                for (int j = 0; j < q.kRegs; ++j) {
                    const int f = sub + G * j;
                    q.r[j] = f < F4 ? ldg4(qv + 4 * f) : make_float4(0.f, 0.f, 0.f, 0.f);
                }
            }
        }
        uint32_t qc[CLay::W];
        int32_t qq = 0;          // this lane's share of the query's code norm
        if (MODE != kCodeNone) {
            code_words<F4, VAR>(JF(qcodes) + (int64_t)qrow * (4 * F4), lane % CLay::G, qc);
#pragma unroll
            for (int j = 0; j < CLay::W; ++j) qq = (int32_t)__dp4a(qc[j], qc[j], (uint32_t)qq);
        }
        for (uint32_t i = lane; i < table.buckets; i += 32) reinterpret_cast<int4 *>(tab)[i] = make_int4(-1, -1, -1, -1);
        __syncwarp();

        beam_t k[PER];
#pragma unroll
        for (int t = 0; t < PER; ++t) k[t] = ~0ull;
        beam_t worst = ~0ull;
        bool lossy = false;
        uint32_t ndc = 0, nexp = 0;

        // Batches of up to 32 ids: first the entry points, then, list by list, the
        // neighbours of the nearest unexpanded entry.  The runner-up's list is loaded
        // with it: it is usually expanded next, and its list is then at hand.
        const int n_seeds = a.seed_mode == kSeedTable ? a.n_seeds : 1;
        int32_t u = 0;                          // the vertex being expanded,
        int nb_at = INT32_MAX;                  // its list from here on
        int32_t n0 = -1, n1 = -1;               // ids 0..63 of the runner-up's list
        int32_t ahead = -1;                     // the runner-up
        int32_t c1 = -1;                        // ids 32..63 of the current list
        for (int s0 = 0;; ) {
            int32_t cand = -1, pf = -1;
            if (s0 < n_seeds) {
                if (a.seed_mode == kSeedTable) {
                    const int32_t *seed_row = JF(seed_row);
                    const int32_t *srow = JF(seed_tab) + (seed_row ? (int64_t)seed_row[qrow] : gi) * a.seed_stride;
                    if (s0 + lane < n_seeds) cand = srow[s0 + lane];
                    if (cand >= JF(n_base)) cand = -1;
                } else if (lane == 0) {
                    cand = a.seed_mode == kSeedSelf ? qrow : JF(seed_const);
                }
                s0 += 32;
            } else if (nb_at < JF(r_in)) {
                const int r_in = JF(r_in);
                cand = nb_at == 32 ? c1 : nb_at + lane < r_in ? JF(adj)[(int64_t)u * r_in + nb_at + lane] : -1;
                nb_at += 32;
            } else {
                int found = -1, second = -1;
                beam_t kf = 0, ks = 0;
#pragma unroll
                for (int t = 0; t < PER; ++t) {
                    unsigned m = __ballot_sync(0xffffffffu, (k[t] & 1ull) == 0 && 32 * t + lane < a.ef);
                    if (found < 0 && m) {
                        found = 32 * t + __ffs(m) - 1;
                        kf = k[t];
                        m &= m - 1u;
                    }
                    if (found >= 0 && second < 0 && m) {
                        second = 32 * t + __ffs(m) - 1;
                        ks = k[t];
                    }
                }
                if (found < 0) break;
                u = (int32_t)(__shfl_sync(0xffffffffu, (uint32_t)kf, found & 31) >> 1);
#pragma unroll
                for (int t = 0; t < PER; ++t)
                    if (found == 32 * t + lane) k[t] |= 1ull;
                ++nexp;
                const int32_t *adj = JF(adj);
                const int r_in = JF(r_in);
                const int32_t *nb = adj + (int64_t)u * r_in;
                cand = n0;
                c1 = n1;
                if (u != ahead) {
                    cand = lane < r_in ? nb[lane] : -1;
                    if (r_in > 32) c1 = lane + 32 < r_in ? nb[lane + 32] : -1;
                }
                nb_at = 32;
                ahead = -1;
                if (second >= 0) {
                    ahead = (int32_t)(__shfl_sync(0xffffffffu, (uint32_t)ks, second & 31) >> 1);
                    const int32_t *nx = adj + (int64_t)ahead * r_in;
                    n0 = lane < r_in ? nx[lane] : -1;
                    if (r_in > 32) n1 = lane + 32 < r_in ? nx[lane + 32] : -1;
                    if (prefetch) pf = n0;
                }
            }
            const bool fresh = EFMAX > 64 && VAR != kLatencyShape && table.tag_shift > 0
                                   ? visit_tags(tab, table.buckets, table.shift, table.tag_shift, cand, cand >= 0, lossy)
                                   : visit(tab, table.buckets / 2, cand, cand >= 0, lossy);
            const unsigned m = __ballot_sync(0xffffffffu, fresh);
            const int c = __popc(m);
            if (fresh) ci[__popc(m & lanemask_lt())] = cand;
            // pf: a neighbour of the entry likely to be expanded next; its row is
            // brought into L2 now so that the next gather finds it there (a hint only)
            if (pf >= 0) {
                const char *pr = MODE == kCodeNone ? reinterpret_cast<const char *>(JF(base)) + (int64_t)pf * (16 * F4)
                                                   : reinterpret_cast<const char *>(JF(codes)) + (int64_t)pf * (4 * F4);
#pragma unroll
                for (int l = 0; l < (MODE == kCodeNone ? 16 : 4) * F4; l += 128) prefetch_l2(pr + l);
            }
            __syncwarp();
            ndc += (uint32_t)c;
            if (MODE == kCodeNone) {
                eval_rows<F4, PER, MODE, VAR>(a, JF(base), ci, c, q, k, worst, lossy, scratch);
            } else {
                const float limit = MODE == kCodeFilter ? code_limit(cp, a.metric, worst) : 0.f;
                const int np = eval_codes<F4, PER, MODE, VAR>(a, JF(codes), ci, c, qc, qq, limit, pass, k, worst, lossy, scratch);
                if (MODE == kCodeFilter) {
                    __syncwarp();
                    eval_rows<F4, PER, MODE, VAR>(a, JF(base), pass, np, q, k, worst, lossy, scratch);
                }
            }
            __syncwarp();   // ci is read before the next batch overwrites it
        }

        if (!early && lane == 0) claim = atomicAdd(a.work, 1);

        // Output: first a.k entries of C (optionally without the query vertex).
        const int32_t self = a.exclude_self ? qrow : -1;
        const int64_t orow = a.out_by_qidx ? qrow : gi;
        int32_t *oid = JF(out_ids) + orow * a.out_stride;
        float *od = (!JOBS && a.out_d) ? a.out_d + orow * a.out_stride : nullptr;
        const int32_t id_offset = JF(id_offset);
        int written = 0;
#pragma unroll
        for (int t = 0; t < PER; ++t) {
            const int32_t id = (int32_t)((uint32_t)k[t] >> 1);
            const bool keep = k[t] != ~0ull && 32 * t + lane < a.ef && id != self;
            const unsigned m = __ballot_sync(0xffffffffu, keep);
            const int pos = written + __popc(m & lanemask_lt());
            if (keep && pos < a.k) {
                oid[pos] = id + id_offset;
                if (od) od[pos] = unorder_bits((uint32_t)(k[t] >> 32));
            }
            written += __popc(m);
        }
        for (int j = written + lane; j < a.k; j += 32) {
            oid[j] = -1;
            if (od) od[j] = FLT_MAX;
        }
        if (!JOBS && lane == 0 && a.out_ndc) a.out_ndc[gi] = (int64_t)ndc;
        ndc_total += ndc;
        nexp_total += nexp;
        __syncwarp();
    }
    if (lane == 0 && a.stats) {
        atomicAdd(&a.stats[0], ndc_total);
        atomicAdd(&a.stats[1], nexp_total);
    }
}

#undef JF

// The visited table of a launch.  A search meets up to 1.2 * ef * r_in different
// vertices (DEEP-like rows, whose lists hardly overlap; SIFT-like ones half of
// that); 1.25 * ef * r_in slots remember them all, and where that many would cost
// resident warps, fewer: 1,536 slots against 4,096 took 24 % off the pivot searches
// of 2 x 500k SIFT-like rows (ef 64) for 0.9 % more evaluations.  Beams over 64 take
// tags, which remember twice as much in the same bytes: 24 a beam entry up to ef 128
// and for lists over 48, else 20 (24 there cost warps: 10k DEEP-like queries, ef 256
// 5.6 ms, 20 4.8).  Evaluations above those of an exact visited set (20k rows), and
// time of 10k queries, with 1,536 or 2,048 ids and as below: DEEP-like R 32, ef 256
// 20.9 -> 2.5 %, 5.1 -> 4.8 ms; embedding-like R 64, ef 128 15.5 -> 8.6 %, 8.9 -> 8.2 ms
// and ef 256 40.4 -> 10.8 %, 20.5 -> 18.2 ms; 24 ids a beam entry: 0.6, 8.3 and 9.5 %, 7.8,
// 9.4 and 45.5 ms.  (FP32 rows only, d = 128, ef 256: 6.2 -> 6.9 ms for 7 % fewer
// evaluations.)  A tag costs some ten instructions more a lookup than an id, so short
// lists keep ids (50k Gaussian rows, R 16, ef 128: 2,048 ids 1.13 ms, tags 1.22, 1,536 ids
// 1.16); so do graphs whose ids need more than 15 bits beside the set.
//
// The latency shape takes up to 8,192 ids for launches that one CTA per SM holds, else
// 6,144, with which two fit: 1,216 queries, ef 256, took two waves of 152 CTAs with more (50k
// Gaussian rows of 8 dimensions, R 24: 1.07 ms, now 0.44; 30k embedding-like rows 6.7, 3.5).
template <int VAR>
TableShape table_shape(int ef, int r_in, int64_t n, int64_t nq) {
    const int most = VAR != kLatencyShape ? (VAR == 1 ? 2048 : 1536) : nq > kLatencyQueries / 2 ? 6144 : 8192;
    const int all = std::max(ef * r_in + ef * r_in / 4, 1024);
    TableShape t = {};
    if (VAR != kLatencyShape && ef > 64 && all > 2560) {
        const int per = ef <= 128 || r_in > 48 ? 24 : 20;
        const int buckets = (std::min(all, per * ef) + 63) / 64 * 8, lg = 31 - __builtin_clz((unsigned)buckets);
        int b = lg + 1;
        while (b < 31 && ((int64_t)1 << b) < n) ++b;
        if (b - lg <= 15) {
            t.buckets = (uint32_t)buckets;
            t.shift = 32 - b;
            t.tag_shift = 32 - b + lg;
            return t;
        }
    }
    const int slots = std::min(all, ef > 64 ? std::max(most, 2048) : most);
    t.buckets = (uint32_t)(slots + 63) / 64 * 16;
    return t;
}

template <int F4, int EFMAX, int MODE, int VAR, bool JOBS>
cudaError_t launch_t(const SearchArgs &a, int prefetch, cudaStream_t st) {
    const TableShape table = table_shape<VAR>(a.ef, a.r_in, a.n_base, a.nq);
    const size_t smem = (size_t)kSearchWarps * warp_smem_bytes(table.buckets, EFMAX, MODE == kCodeFilter ? F4 : 0);
    auto kern = search_kernel<F4, EFMAX, MODE, VAR, JOBS>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem);
    if (e != cudaSuccess) return e;
    // the visited tables live in shared memory: ask for the largest carveout
    cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    cudaFuncAttributes fa;
    e = cudaFuncGetAttributes(&fa, kern);
    if (e != cudaSuccess) return e;
    int dev = 0, sms = 0, smem_sm = 0, regs_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    cudaDeviceGetAttribute(&regs_sm, cudaDevAttrMaxRegistersPerMultiprocessor, dev);
    int per_sm = smem_sm / (int)(fa.sharedSizeBytes + smem + 1024);
    const int by_regs = regs_sm / ((fa.numRegs > 0 ? fa.numRegs : 64) * kSearchWarps * 32);
    if (by_regs < per_sm) per_sm = by_regs;
    if (per_sm > 2048 / (kSearchWarps * 32)) per_sm = 2048 / (kSearchWarps * 32);
    if (per_sm < 1) per_sm = 1;
    int64_t want = (a.nq + kSearchWarps - 1) / kSearchWarps;
    int64_t grid = (int64_t)sms * per_sm;
    if (want < grid) grid = want < 1 ? 1 : want;
    kern<<<(unsigned)grid, kSearchWarps * 32, smem, st>>>(a, table, prefetch);
    note_launches(1);
    return cudaGetLastError();
}

template <int F4, int EFMAX, int MODE, bool JOBS>
cudaError_t launch_var(const SearchArgs &a, int var, cudaStream_t st) {
    const int pf = (var >> 1) & 1;
    if (a.nq <= kLatencyQueries) return launch_t<F4, EFMAX, MODE, kLatencyShape, JOBS>(a, pf, st);
    if constexpr (MODE != kCodeExact)   // (code rows alone: one shape)
        if (var & 1) return launch_t<F4, EFMAX, MODE, 1, JOBS>(a, pf, st);
    return launch_t<F4, EFMAX, MODE, 0, JOBS>(a, pf, st);
}

template <int F4, int MODE, bool JOBS>
cudaError_t launch_ef(const SearchArgs &a, int var, cudaStream_t st) {
    if (a.ef <= 32) return launch_var<F4, 32, MODE, JOBS>(a, var, st);
    if (a.ef <= 64) return launch_var<F4, 64, MODE, JOBS>(a, var, st);
    if (a.ef <= 128) return launch_var<F4, 128, MODE, JOBS>(a, var, st);
    return launch_var<F4, 256, MODE, JOBS>(a, var, st);
}

template <bool JOBS>
cudaError_t launch_plain(const SearchArgs &a, int var, cudaStream_t st) {
    switch (a.dim) {
        case 8: return launch_ef<2, kCodeNone, JOBS>(a, var, st);
        case 16: return launch_ef<4, kCodeNone, JOBS>(a, var, st);
        case 32: return launch_ef<8, kCodeNone, JOBS>(a, var, st);
        case 64: return launch_ef<16, kCodeNone, JOBS>(a, var, st);
        case 96: return launch_ef<24, kCodeNone, JOBS>(a, var, st);
        case 128: return launch_ef<32, kCodeNone, JOBS>(a, var, st);
        case 256: return launch_ef<64, kCodeNone, JOBS>(a, var, st);
        case 768: return launch_ef<192, kCodeNone, JOBS>(a, var, st);
        default: return cudaErrorInvalidValue;
    }
}

template <bool JOBS>
cudaError_t launch_filter(const SearchArgs &a, int var, cudaStream_t st) {
    switch (a.dim) {
        case 64: return launch_ef<16, kCodeFilter, JOBS>(a, var, st);
        case 96: return launch_ef<24, kCodeFilter, JOBS>(a, var, st);
        case 128: return launch_ef<32, kCodeFilter, JOBS>(a, var, st);
        case 256: return launch_ef<64, kCodeFilter, JOBS>(a, var, st);
        case 768: return launch_ef<192, kCodeFilter, JOBS>(a, var, st);
        default: return cudaErrorInvalidValue;
    }
}

template <bool JOBS>
cudaError_t launch_exact(const SearchArgs &a, int var, cudaStream_t st) {
    switch (a.dim) {   // 256 * 255^2 < 2^24: every distance is exact in FP32
        case 64: return launch_ef<16, kCodeExact, JOBS>(a, var, st);
        case 96: return launch_ef<24, kCodeExact, JOBS>(a, var, st);
        case 128: return launch_ef<32, kCodeExact, JOBS>(a, var, st);
        case 256: return launch_ef<64, kCodeExact, JOBS>(a, var, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace
}  // namespace rnsm
