// K1: batched AKNN beam search (Algorithm 1, Section 2.2), one warp per query:
// launch shapes and their autotuner; the kernel is in search_impl.cuh.
//
// Per warp: the candidate set C sorted in registers (64-bit keys of distance, id
// and the expanded flag), a visited table in shared memory, and the neighbours'
// rows gathered with 128-bit loads: first their codes (codes.cu), then, where
// those do not settle it, their FP32 rows, of which a group of G lanes covers one
// (lane s of the group reads float4 s, s+G, ...), 32/G rows per step.
//
// Semantics match Algorithm 1 exactly: repeatedly expand the nearest
// unexpanded entry, evaluate every neighbour not evaluated before, keep the
// best ef by (distance, id).  Inserting a whole neighbourhood and truncating
// to ef leaves the same set as inserting one neighbour at a time.  The visited
// table is exact until a set of it is full; from then on it may forget, which
// cannot change the result because an evaluated vertex outside C is worse
// than the worst entry of C (and that bound only tightens) while vertices
// inside C are found there before insertion.
//
// What bounds it: the instructions of an expansion.  2 x 500k SIFT-like rows, S1 +
// S4 + S5, before (C and merge by ranks in shared memory, FP32 rows, a hash probed
// slot by slot): 7.2 + 7.7 + 8.7 ms at 76 % of L2 throughput; now 4.1 + 4.7 + 5.6
// ms at 80 % of the issue slots and 31 % of L2 throughput.  300k DEEP-like rows:
// 4.3 + 8.2 + 12.3 -> 3.2 + 4.5 + 7.6 ms; 60k embedding-like rows of 768:
// 4.6 + 12.7 + 16.7 -> 2.8 + 5.3 + 9.6 ms; 16 queries, ef 128, on 100k DEEP-like
// rows: 1.9 -> 0.40 ms.
#include <float.h>
#include <stdlib.h>

#include <map>
#include <mutex>
#include <utility>

#include "internal.h"

namespace rnsm {

namespace {

cudaError_t launch_dim_any(const SearchArgs &a, int var, cudaStream_t st) {
    // few queries: each warp's chain of dependent loads decides, and the filter's
    // second gather would lengthen it
    const int mode = a.code_mode == kCodeFilter && a.nq <= kLatencyQueries ? kCodeNone : a.code_mode;
    switch (mode) {
        case kCodeExact: return a.jobs ? launch_search_jobs_exact(a, var, st) : launch_search_exact(a, var, st);
        case kCodeFilter: return a.jobs ? launch_search_jobs_filter(a, var, st) : launch_search_filter(a, var, st);
        default: return a.jobs ? launch_search_jobs_plain(a, var, st) : launch_search_plain(a, var, st);
    }
}

// The queries [q0, q1) of a launch as a launch of their own.
SearchArgs subrange(const SearchArgs &a, int64_t q0, int64_t q1) {
    SearchArgs b = a;
    b.q0 = a.q0 + q0;
    b.nq = q1 - q0;
    return b;
}

// Autotuner: the first launch of a (dim, beam, seed mode) shape with at least
// kTuneChunks * kTuneMinChunk queries runs as kTuneChunks consecutive chunks
// spread over its whole query list, the variants taking turns (the order
// rotating every round), each chunk timed with CUDA events on the launching
// stream and its distance computations counted.  The variant with the least
// time per distance computation is kept for later launches of that shape.
// Every query runs once, with final results (all variants compute the same
// beams); normalising by the distance count makes chunks of different
// difficulty comparable, and spreading the chunks over the list keeps the
// comparison representative when the queries come in locality order.
constexpr int kVariants = 4;   // search_impl.cuh: shape, prefetch
constexpr int kTuneChunks = 4 * kVariants;
constexpr int64_t kTuneMinChunk = 4000;
struct TuneKey {
    int dim, efmax, seed_mode, code_mode;
    bool operator<(const TuneKey &o) const {
        if (code_mode != o.code_mode) return code_mode < o.code_mode;
        return dim != o.dim ? dim < o.dim : efmax != o.efmax ? efmax < o.efmax : seed_mode < o.seed_mode;
    }
};
std::mutex g_tune_mu;
std::map<TuneKey, int> g_tuned;

int efmax_of(int ef) { return ef <= 32 ? 32 : ef <= 64 ? 64 : ef <= 128 ? 128 : 256; }

int forced_variant() {
    const char *force = getenv("RNSM_SEARCH_VARIANT");
    return force && force[0] >= '0' && force[0] < '0' + kVariants ? force[0] - '0' : -1;
}

// Before a shape is tuned (and for launches too small to tune): shape 1 where a
// lane's share of a row is six float4 and few rows are in flight otherwise.
// Embedding-like rows (768, filtered): S4 10.5 -> 5.6 ms, S5 15.0 -> 10.1 ms on
// 3 x 20k; DEEP-like rows (96, FP32 only): S4 6.7 -> 5.4, S5 9.4 -> 9.1 ms on
// 300k; SIFT-like rows (128, FP32 only) S5 8.6 -> 11.6 ms on 2 x 500k.  The dimensions
// with no merge behind them, 20k queries, ef 32 / 64 / 128, shape 0 and 1: 64 filtered 0.93 /
// 1.49 / 2.96 and 1.11 / 1.82 / 3.50 ms, FP32 only 0.95 / 1.59 / 3.22 and 0.91 / 1.50 / 3.27;
// 256 filtered 1.97 / 3.31 / 6.76 and 2.06 / 3.60 / 6.49, FP32 only 2.94 / 4.95 / 8.76 and 2.91 /
// 4.85 / 9.10.  (Filtered against FP32 only: 64 0.92 / 1.49 / 2.95 and 0.91 / 1.52 / 3.14 ms, 128
// 1.38 / 2.33 / 4.25 and 1.86 / 3.14 / 5.66.)
int default_variant(int dim, int code_mode) {
    return dim == 768 || (dim == 96 && code_mode == kCodeNone) ? 1 : 0;
}

}  // namespace

bool search_would_tune(int dim, int ef, int seed_mode, int code_mode, int64_t nq) {
    if (forced_variant() >= 0 || nq < kTuneChunks * kTuneMinChunk) return false;
    std::lock_guard<std::mutex> lk(g_tune_mu);
    return g_tuned.find({dim, efmax_of(ef), seed_mode, code_mode}) == g_tuned.end();
}

cudaError_t launch_search(const SearchArgs &a, cudaStream_t st) {
    if (a.nq <= 0) return cudaSuccess;
    if (!search_dim_supported(a.dim)) return cudaErrorInvalidValue;
    const int forced = forced_variant();
    if (forced >= 0) return launch_dim_any(a, forced, st);
    const TuneKey key{a.dim, efmax_of(a.ef), a.seed_mode, a.code_mode};
    int var = -1;
    const int first = default_variant(a.dim, a.code_mode);
    {
        std::lock_guard<std::mutex> lk(g_tune_mu);
        auto it = g_tuned.find(key);
        if (it != g_tuned.end()) var = it->second;
    }
    if (var >= 0 || a.nq < kTuneChunks * kTuneMinChunk) return launch_dim_any(a, var >= 0 ? var : first, st);
    // NDC of each chunk: the caller's statistics counter, read around the chunk
    static unsigned long long *own_stats[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    unsigned long long *cnt = a.stats;
    if (!cnt) {
        if (dev >= 64) return launch_dim_any(a, first, st);
        if (!own_stats[dev] && cudaMalloc(&own_stats[dev], 2 * sizeof(unsigned long long)) != cudaSuccess)
            return launch_dim_any(a, first, st);
        cnt = own_stats[dev];
    }
    double ms_of[kVariants] = {}, ndc_of[kVariants] = {};
    cudaEvent_t e0, e1;
    if (cudaEventCreate(&e0) != cudaSuccess) return launch_dim_any(a, first, st);
    if (cudaEventCreate(&e1) != cudaSuccess) {
        cudaEventDestroy(e0);
        return launch_dim_any(a, first, st);
    }
    cudaError_t err = cudaSuccess;
    unsigned long long before = 0, after = 0;
    for (int c = 0; c < kTuneChunks && err == cudaSuccess; ++c) {
        const int v = (c + c / kVariants) % kVariants;
        SearchArgs sl = subrange(a, a.nq * c / kTuneChunks, a.nq * (c + 1) / kTuneChunks);
        sl.stats = cnt;
        err = cudaMemcpyAsync(&before, cnt, sizeof(before), cudaMemcpyDeviceToHost, st);
        if (err == cudaSuccess) err = cudaMemsetAsync(a.work, 0, sizeof(int32_t), st);
        if (err == cudaSuccess) err = cudaEventRecord(e0, st);
        if (err == cudaSuccess) err = launch_dim_any(sl, v, st);
        if (err == cudaSuccess) err = cudaEventRecord(e1, st);
        if (err == cudaSuccess) err = cudaMemcpyAsync(&after, cnt, sizeof(after), cudaMemcpyDeviceToHost, st);
        if (err == cudaSuccess) err = cudaStreamSynchronize(st);
        float ms = 0.f;
        if (err == cudaSuccess) err = cudaEventElapsedTime(&ms, e0, e1);
        ms_of[v] += ms;
        ndc_of[v] += (double)(after - before);
    }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if (err != cudaSuccess) return err;
    int best = 0;
    for (int v = 1; v < kVariants; ++v)
        if (ms_of[v] * ndc_of[best] < ms_of[best] * ndc_of[v]) best = v;
    std::lock_guard<std::mutex> lk(g_tune_mu);
    g_tuned[key] = best;
    return cudaSuccess;
}

bool search_dim_supported(int dim) {
    switch (dim) {
        case 8: case 16: case 32: case 64: case 96: case 128: case 256: case 768: return true;
        default: return false;
    }
}

}  // namespace rnsm
