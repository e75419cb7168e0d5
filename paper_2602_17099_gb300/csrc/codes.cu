// Coded rows: a byte per dimension beside the FP32 rows, for the searches.
//
// A search evaluates some 15 to 45 vertices for every one it keeps near the
// end; each costs a gathered FP32 row (4 bytes a dimension) and two FP32
// operations a dimension.  With x ~ lo + s * c, c in 0..255, the squared
// distance of two code rows, s^2 * S with S = sum (c_x - c_q)^2 an exact
// integer, comes from a quarter of the bytes and dp4a, and
//     |  ||x - q|| - s * sqrt(S)  |  <=  e_x + e_q,   e = ||x - (lo + s * c)||,
// so most candidates are known to lie beyond the beam's worst entry before
// their FP32 row is touched.  Only the others get their FP32 distance, by which
// alone everything is decided: the results are those of the FP32 search.
// Rows of integers that span at most 255 (SIFT) have s = 1 and e = 0: S is the
// squared distance itself, and no FP32 row is needed (kCodeExact).
#include <float.h>

#include "internal.h"

namespace rnsm {

namespace {

__device__ __forceinline__ uint32_t order_key(float f) {
    const uint32_t b = __float_as_uint(f);
    return b ^ ((uint32_t)((int32_t)b >> 31) | 0x80000000u);
}
__device__ __forceinline__ float order_value(uint32_t u) {
    return __uint_as_float((u & 0x80000000u) ? u ^ 0x80000000u : ~u);
}

// Block-wide reductions of the passes below: one atomic per block and value
// (one per warp: 0.28 ms more on 300k rows of 96, all to the same words).
__device__ __forceinline__ float block_max(float v, float *sh) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
    const int warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    __syncthreads();
    if ((threadIdx.x & 31) == 0) sh[warp] = v;
    __syncthreads();
    for (int w = 0; w < nw; ++w) v = fmaxf(v, sh[w]);
    return v;
}

// Finite check, smallest and largest component and whether all are integers,
// in the one pass that the finite check (of the first `checked` segments) needs
// anyway.
__global__ void __launch_bounds__(256) code_scan_kernel(const SegTable t, int dim, int checked, CodeStats *s,
                                                        int32_t *err) {
    __shared__ float sh[8];
    float lo = INFINITY, hi = -INFINITY;
    bool frac = false, bad = false;
    for (int g = 0; g < t.m; ++g) {
        const float4 *v = reinterpret_cast<const float4 *>(t.base[g]);
        const int64_t count4 = (t.off[g + 1] - t.off[g]) * (dim / 4);
        for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < count4;
             i += (int64_t)gridDim.x * blockDim.x) {
            const float4 x = __ldg(v + i);
            lo = fminf(lo, fminf(fminf(x.x, x.y), fminf(x.z, x.w)));
            hi = fmaxf(hi, fmaxf(fmaxf(x.x, x.y), fmaxf(x.z, x.w)));
            frac = frac || rintf(x.x) != x.x || rintf(x.y) != x.y || rintf(x.z) != x.z || rintf(x.w) != x.w;
            bad = bad || (g < checked && (!isfinite(x.x) || !isfinite(x.y) || !isfinite(x.z) || !isfinite(x.w)));
        }
    }
    lo = -block_max(-lo, sh);
    hi = block_max(hi, sh);
    frac = __syncthreads_or(frac);
    bad = __syncthreads_or(bad);
    if (threadIdx.x == 0) {
        if (lo <= hi) {
            atomicMax(&s->omin_inv, ~order_key(lo));
            atomicMax(&s->omax, order_key(hi));
        }
        if (frac) atomicOr(&s->fraction, 1);
        if (bad) atomicOr(err, 2);
    }
}

// lo and s of the scanned rows; s = 0: no codes (a range that is empty, not
// finite, or so large or small that the bounds below could leave FP32's range;
// or only exact codes are wanted).
__device__ __forceinline__ void code_grid(const CodeStats *st, float &lo, float &s) {
    const float a = order_value(~st->omin_inv), b = order_value(st->omax);
    const float range = b - a;
    lo = a;
    s = 0.f;
    if (!st->fraction && range <= 255.f && fabsf(a) <= 65536.f) s = 1.f;
    else if (st->exact_only) s = 0.f;
    else if (range > 1e-12f && range < 1e12f && fabsf(a) < 1e12f) s = range / 255.f;
}

// A warp per row: its codes, and the largest squared residual and squared norm.
__global__ void __launch_bounds__(256) code_rows_kernel(const SegTable t, int dim, uint8_t *codes, CodeStats *st) {
    __shared__ float sh[8];
    const int lane = threadIdx.x & 31;
    const int64_t w0 = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
    const int64_t n = t.off[t.m];
    float lo, s;
    code_grid(st, lo, s);
    if (s == 0.f) return;
    const float inv = 1.f / s;
    float e_max = 0.f, n_max = 0.f;
    int g = 0;
    for (int64_t r = w0; r < n; r += nw) {
        while (r >= t.off[g + 1]) ++g;
        const float4 *row = reinterpret_cast<const float4 *>(t.base[g] + (r - t.off[g]) * dim);
        float e = 0.f, nn = 0.f;
        for (int f = lane; f < dim / 4; f += 32) {
            const float4 x = __ldg(row + f);
            uint32_t w = 0;
            const float xs[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float y = xs[j] - lo;
                const float c = fminf(fmaxf(rintf(y * inv), 0.f), 255.f);
                const float d = fmaf(-s, c, y);
                e = fmaf(d, d, e);
                nn = fmaf(xs[j], xs[j], nn);
                w |= (uint32_t)c << (8 * j);
            }
            reinterpret_cast<uint32_t *>(codes + r * dim)[f] = w;
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            e += __shfl_xor_sync(0xffffffffu, e, o);
            nn += __shfl_xor_sync(0xffffffffu, nn, o);
        }
        e_max = fmaxf(e_max, e);
        n_max = fmaxf(n_max, nn);
    }
    e_max = block_max(e_max, sh);
    n_max = block_max(n_max, sh);
    if (threadIdx.x == 0) {
        // non-negative floats order as their bits
        if (e_max > 0.f) atomicMax(&st->err2, __float_as_uint(e_max));
        atomicMax(&st->norm2, __float_as_uint(n_max));
    }
}

constexpr int kSampleDim = 128;   // the widest rows that the coded prune takes

// Sample k of the prunes: how many of its kept rows leave a test open.  The greedy walk
// over up to 32 candidates of owner k's list with FP32 distances; a test "does s
// occlude c" is open where sqrt(d(s, c)) lies within err of sqrt(d(v, c) / alpha), as
// limits_of in prune_code.cu has it but for the rounding terms.
constexpr int kSampleThreads = 256, kSampleRows = 32;
constexpr int kSamplePairs = (kSampleRows + 1) * kSampleRows / 2;
struct SampleSmem {
    float4 row[(kSampleRows + 1) * (kSampleDim / 4 + 1)];   // stride 16 (mod 128) bytes; the last: the owner
    float dist[kSampleRows + 1][kSampleRows + 1];
    int32_t id[kSampleRows + 1];
    int32_t at[kSampleRows];        // candidate at each position of the order
};
// By the first warp: the owner's and its candidates' ids (-1: none).
__device__ __forceinline__ void sample_list(SampleSmem &s, const SegTable &t, const CodeLists &l, int k) {
    const int lane = threadIdx.x;
    const int64_t n = t.off[t.m];
    int64_t v = (l.owners ? l.n_owners : n) * k / kCodeSamples, at = v;
    int g = 0;
    if (l.owners) {
        v = l.owners[v];
        if (l.by_id) at = v;
    } else {
        while (v >= t.off[g + 1]) ++g;
        at = v - t.off[g];
    }
    const int len = l.rows[g] && v >= 0 && v < n ? l.len[g] : 0;
    int32_t c = -1;
    if (lane < len) c = l.rows[g][at * len + (len > kSampleRows ? (int64_t)lane * len / kSampleRows : lane)];
    c = c >= 0 && c < t.off[g + 1] - t.off[g] ? c + (int32_t)t.off[g] : -1;   // (not checked yet)
    const unsigned same = __match_any_sync(0xffffffffu, c);   // (every lane takes part)
    if (c == v || __ffs(same) - 1 != lane) c = -1;
    s.id[lane] = c;
    if (lane == 0) s.id[kSampleRows] = len > 0 ? (int32_t)v : -1;
}
__device__ __forceinline__ void sample_prune(SampleSmem &s, const SegTable &t, int dim, float alpha, float err, int &steps,
                                             int &open_steps) {
    const int tid = threadIdx.x, lane = tid & 31, f4 = dim / 4, stride = kSampleDim / 4 + 1;
    for (int u = tid; u < (kSampleRows + 1) * f4; u += kSampleThreads) {
        const int r = u / f4, f = u - r * f4;
        if (s.id[r] >= 0) s.row[r * stride + f] = ldg4(seg_row(t, s.id[r], dim) + 4 * f);
    }
    __syncthreads();
    for (int u = tid; u < kSamplePairs; u += kSampleThreads) {   // the pairs of 33 rows, a triangle folded to rows of 33
        const int r = u / (kSampleRows + 1), q = u - r * (kSampleRows + 1);
        const int m = kSampleRows / 2 + 1 + r;   // of row 15 - r; the others of row 16 + r
        const int a = q < m ? kSampleRows / 2 - 1 - r : kSampleRows / 2 + r, b = a + 1 + (q < m ? q : q - m);
        if (s.id[a] >= 0 && s.id[b] >= 0) {
            float d = 0.f;
            for (int f = 0; f < f4; ++f) d = l2_acc(d, s.row[a * stride + f], s.row[b * stride + f]);
            s.dist[a][b] = s.dist[b][a] = d;
        }
    }
    __syncthreads();
    if (tid >= kSampleRows) return;
    // lane r: the candidate at position r of the (distance, slot) order, none: infinity
    float dv = s.id[lane] >= 0 ? s.dist[kSampleRows][lane] : INFINITY;
    int rank = 0;
#pragma unroll
    for (int j = 0; j < 32; ++j) {
        const float o = __shfl_sync(0xffffffffu, dv, j);
        rank += o < dv || (o == dv && j < lane);
    }
    s.at[lane] = 0;
    __syncwarp();
    s.at[rank] = lane;
    __syncwarp();
    const int mine = s.at[lane], last = __popc(__ballot_sync(0xffffffffu, s.id[lane] >= 0));
    dv = s.dist[kSampleRows][mine];
    const float root = sqrtf(dv / alpha);
    unsigned occluders = 0u, open = 0u;   // positions before this one
#pragma unroll 8
    for (int r = 0; r < 32; ++r) {
        const float d = s.dist[s.at[r]][mine];
        if (fmaf(alpha, d, -dv) <= 0.f) occluders |= 1u << r;
        if (fabsf(sqrtf(d) - root) <= err) open |= 1u << r;
    }
    const unsigned before = lane < last ? (1u << lane) - 1u : 0u;
    occluders &= before;
    unsigned kept = 0u;
#pragma unroll
    for (int r = 0; r < 32; ++r) {
        const unsigned o = __shfl_sync(0xffffffffu, occluders, r);
        if (r < last && (o & kept) == 0u) kept |= 1u << r;
    }
    // tested by the kept rows up to the first that occludes it
    const unsigned by = occluders & kept, tested = before & kept & (by ? (by ^ (by - 1u)) : ~0u);
    steps = __popc(__reduce_or_sync(0xffffffffu, tested));
    open_steps = __popc(__reduce_or_sync(0xffffffffu, tested & open));
}

// The constants.  err: e_x + e_q of any two rows, with the roundings of y = x - lo
// (half an ulp of the range a component), of the residual and of its sum taken in.
// useful: on sampled pairs of rows far apart in the table the bound's slack is small
// against their distance.  Near neighbours are a few times closer than such pairs; with
// the slack under kSlack of the distance most candidates of a converged beam are settled
// by their codes (DEEP-like rows 0.016, embeddings 0.022), with a lone component much
// larger than the rest few would be.  The prunes compare neighbours with each other, and
// are sampled for themselves (lists; L2 only).  A block a sample, the last one done
// writes the result and leaves the sample counts as it found them, for another call.
constexpr float kSlack = 0.04f;
__global__ void __launch_bounds__(kSampleThreads) code_params_kernel(const __grid_constant__ SegTable t, int dim, int metric,
                                                                     const __grid_constant__ CodeLists lists,
                                                                     CodeStats *st, CodeParams *p) {
    __shared__ SampleSmem smem;
    __shared__ int last;
    const int lane = threadIdx.x & 31, k = blockIdx.x;
    const int64_t n = t.off[t.m];
    const bool listed = metric == 0 && dim <= kSampleDim && lists.alpha > 0.f;
    if (listed && threadIdx.x < 32) sample_list(smem, t, lists, k);
    float lo, s;
    code_grid(st, lo, s);
    const bool exact = s == 1.f && !st->fraction;
    const float range = order_value(st->omax) - order_value(~st->omin_inv);
    const float err = exact ? 0.f : 2.f * (1.001f * sqrtf(__uint_as_float(st->err2)) + 1.2e-7f * sqrtf((float)dim) * range);
    if (threadIdx.x >= 32 && threadIdx.x < 64) {   // the pair, by the second warp
        const int64_t a = n * k / kCodeSamples, b = (a + n / 2 + k) % n;
        const float *x = seg_row(t, (int32_t)a, dim), *y = seg_row(t, (int32_t)b, dim);
        float d = 0.f, nn = 0.f;
        for (int j = lane; j < dim; j += 32) {
            const float u = x[j], v = y[j];
            d = fmaf(u - v, u - v, d);
            nn = fmaf(u, u, fmaf(v, v, nn));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            d += __shfl_xor_sync(0xffffffffu, d, o);
            nn += __shfl_xor_sync(0xffffffffu, nn, o);
        }
        if (lane == 0) {
            st->pair_d2[k] = d;
            st->pair_norm2[k] = nn;
            __threadfence();
        }
    }
    int steps = 0, open_steps = 0;
    __syncthreads();
    if (listed && !exact && s > 0.f && smem.id[kSampleRows] >= 0)
        sample_prune(smem, t, dim, lists.alpha, err, steps, open_steps);
    __syncthreads();
    if (threadIdx.x == 0) {
        if (steps) {
            atomicAdd(&st->steps, steps);
            atomicAdd(&st->open_steps, open_steps);
        }
        __threadfence();
        last = atomicAdd(&st->done, 1) == kCodeSamples - 1;
    }
    __syncthreads();
    if (threadIdx.x >= 32 || !last) return;
    __threadfence();
    static_assert(kCodeSamples == 64, "two samples a lane");
    float d2 = __ldcg(&st->pair_d2[lane]) + __ldcg(&st->pair_d2[lane + 32]);
    float nn = __ldcg(&st->pair_norm2[lane]) + __ldcg(&st->pair_norm2[lane + 32]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        d2 += __shfl_xor_sync(0xffffffffu, d2, o);
        nn += __shfl_xor_sync(0xffffffffu, nn, o);
    }
    if (lane != 0) return;
    d2 /= kCodeSamples;
    nn /= kCodeSamples;
    p->scale = s;
    p->inv_scale = s > 0.f ? 1.f / s : 0.f;
    p->exact = exact;
    p->err = err;
    p->norm2 = 1.0001f * __uint_as_float(st->norm2);
    const float gap = metric == 0 ? 0.f : 2.f * p->norm2 - nn;   // code_limit's slack at inner product
    p->useful = s > 0.f && p->err <= kSlack * sqrtf(d2) && gap <= kSlack * d2;
    p->steps = atomicExch(&st->steps, 0);
    p->open_steps = atomicExch(&st->open_steps, 0);
    st->done = 0;
}

}  // namespace

bool codes_dim_ok(int dim) { return dim == 64 || dim == 96 || dim == 128 || dim == 256 || dim == 768; }

cudaError_t launch_code_scan(const SegTable &t, int32_t dim, int32_t checked, CodeStats *s, int32_t *err,
                             cudaStream_t st) {
    int64_t g = (t.off[t.m] * (dim / 4) + 1023) / 1024;
    if (g > 152 * 8) g = 152 * 8;
    code_scan_kernel<<<(unsigned)(g < 1 ? 1 : g), 256, 0, st>>>(t, dim, checked, s, err);
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_code_rows(const SegTable &t, int32_t dim, uint8_t *codes, CodeStats *s, cudaStream_t st) {
    int64_t g = (t.off[t.m] + 7) / 8;
    if (g > 152 * 8) g = 152 * 8;
    code_rows_kernel<<<(unsigned)(g < 1 ? 1 : g), 256, 0, st>>>(t, dim, codes, s);
    note_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_code_params(const SegTable &t, int32_t dim, int32_t metric, const CodeLists &lists, CodeStats *s,
                               CodeParams *p, cudaStream_t st) {
    code_params_kernel<<<kCodeSamples, kSampleThreads, 0, st>>>(t, dim, metric, lists, s, p);
    note_launches(1);
    return cudaGetLastError();
}

}  // namespace rnsm
