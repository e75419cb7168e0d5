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
// finite, or so large or small that the bounds below could leave FP32's range).
__device__ __forceinline__ void code_grid(const CodeStats *st, float &lo, float &s) {
    const float a = order_value(~st->omin_inv), b = order_value(st->omax);
    const float range = b - a;
    lo = a;
    s = 0.f;
    if (!st->fraction && range <= 255.f && fabsf(a) <= 65536.f) s = 1.f;
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

// The search's constants.  err: e_x + e_q of any two rows, with the roundings
// of y = x - lo (half an ulp of the range a component), of the residual and of
// its sum taken in.  useful: on kPairs pairs of rows far apart in the table the
// bound's slack is small against their distance.  Near neighbours are a few
// times closer than such pairs; with the slack under kSlack of the distance most
// candidates of a converged beam are settled by their codes (DEEP-like rows
// 0.016, embeddings 0.022), with a lone component much larger than the rest few
// would be.
constexpr int kPairs = 64;
constexpr float kSlack = 0.04f;
__global__ void __launch_bounds__(1024) code_final_kernel(const SegTable t, int dim, int metric, const CodeStats *st,
                                                          CodeParams *p) {
    __shared__ float sd[kPairs], sn[kPairs];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int64_t n = t.off[t.m];
    for (int k = warp; k < kPairs; k += 32) {
        const int64_t a = (int64_t)((double)n * k / kPairs), b = (a + n / 2 + k) % n;
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
            sd[k] = d;
            sn[k] = nn;
        }
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    float d2 = 0.f, nn = 0.f;
    for (int k = 0; k < kPairs; ++k) {
        d2 += sd[k] / kPairs;
        nn += sn[k] / kPairs;
    }
    float lo, s;
    code_grid(st, lo, s);
    p->scale = s;
    p->inv_scale = s > 0.f ? 1.f / s : 0.f;
    p->exact = s == 1.f && !st->fraction;
    const float range = order_value(st->omax) - order_value(~st->omin_inv);
    const float e = 1.001f * sqrtf(__uint_as_float(st->err2)) + 1.2e-7f * sqrtf((float)dim) * range;
    p->err = p->exact ? 0.f : 2.f * e;
    p->norm2 = 1.0001f * __uint_as_float(st->norm2);
    const float gap = metric == 0 ? 0.f : 2.f * p->norm2 - nn;   // code_limit's slack at inner product
    p->useful = s > 0.f && p->err <= kSlack * sqrtf(d2) && gap <= kSlack * d2;
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

cudaError_t launch_code_rows(const SegTable &t, int32_t dim, int32_t metric, uint8_t *codes, CodeStats *s,
                             CodeParams *p, cudaStream_t st) {
    int64_t g = (t.off[t.m] + 7) / 8;
    if (g > 152 * 8) g = 152 * 8;
    code_rows_kernel<<<(unsigned)(g < 1 ? 1 : g), 256, 0, st>>>(t, dim, codes, s);
    code_final_kernel<<<1, 1024, 0, st>>>(t, dim, metric, s, p);
    note_launches(2);
    return cudaGetLastError();
}

}  // namespace rnsm
