// The occlusion prune over coded rows (codes.cu): L2, d = 64, 96 or 128, pools of at
// most 64 raw candidates; in FP32 mode, and in the tile modes too from the owner count
// that prune_route.cu gives.  Where sampled lists show that the codes would leave many
// tests open (rows in tight clusters) the call does not use them (api.cu, code_prunes).
//
// What bounds the FP32 walk (prune.cu) is that a row of 128 floats a thread leaves
// twelve warps per SM, each waiting on shared memory and barriers.  A coded row is
// 32 words: one warp takes an owner alone, two rows a lane, without any barrier, and
// a pair costs 32 dp4a (norms are computed once) instead of 128 packed FP32
// operations.
//
// Exact (integers spanning up to 255, the codes are the rows): every distance is an
// integer below 2^24, the same that the FP32 chain gives.  Filter (other rows): the
// order comes from FP32 distances to the owner, and a test "does s occlude c" is
// settled by the code distance where its bound allows (limits_of; all but some 2 in
// 1,000 on DEEP-like pools), else by the FP32 distance.  Either way the decisions are
// those of the FP32 kernels.
//
// 2 x 500k SIFT-like rows (exact, d = 128): S6 13.3 -> 2.40 ms, S7 9.7 -> 2.43 ms
// (twenty warps per SM; 16 with registers to spare: 2.47 ms).  DEEP-like rows
// (filter, d = 96): 100k owners, pools of 64, 2.82 -> 1.16 ms (16 warps per SM; 20 with
// spills: 1.15, and a graph build 8 % slower), 1.6 M reverse edges into 150k lists
// 2.70 -> 1.98 ms.
//
// Per owner (one warp): the rows by cp.async into shared memory; every lane its
// two candidates' distances to the owner; positions by counting (64-bit keys of
// distance and id); each lane its two positions' rows into registers; then the
// greedy walk kept row by kept row: the lowest open position is kept, its row is
// read as a broadcast, and the positions after it that it occludes close.
#include "internal.h"

namespace rnsm {

namespace {

constexpr int kCodeWarps = 4;
constexpr int kPool = 64;

template <int W, bool kExact>   // words of a row: 16, 24, 32 (d = 64, 96, 128)
struct CodePool {
    static constexpr int kStride = W + 4;   // words; 8 lanes' 16-byte reads fall on 32 banks
    uint32_t rows[kPool * kStride];
    uint32_t owner[W];                 // the owner's codes
    unsigned long long key[kPool];     // raw order
    unsigned long long order[kPool];   // position order
    int32_t norm[kPool];
    int32_t id[kPool];
    int32_t slot[kPool];               // filter: raw slot of each position
    float4 vrow[kExact ? 1 : W];       // filter: the owner's FP32 row
    const float *rptr[kExact ? 1 : kPool];   // filter: FP32 row of each slot, null: none
};

template <int W, bool kExact>
constexpr int code_blocks() { return (W == 32 ? 5 : W == 24 ? 6 : 8) - (kExact ? 0 : 2); }

// The FP32 distance of two rows by id: the few tests that the codes leave open.  Not
// inlined: its loads would cost the walk registers, and with them warps.
template <int W>
__device__ __noinline__ float far_dist(const SegTable &t, int32_t a, int32_t b) {
    return prune_dist(seg_row(t, a, 4 * W), seg_row(t, b, 4 * W), 4 * W, 0);
}

// Code distances up to `yes` mean that a kept row occludes a candidate at FP32
// distance dv from the owner (alpha * d <= dv), those above `no` that it does not.
// With d the rows' distance, |sqrt(d) - s sqrt(S)| <= err; the FP32 chain is off by
// less than 1e-5 of d at 128 dimensions, and 2e-4 of sqrt(dv / alpha) on either side
// covers it and the roundings here.
struct Limits {
    float yes, no;
};
__device__ __forceinline__ Limits limits_of(float dv, float alpha, float err, float inv_scale) {
    const float t = sqrtf(dv / alpha);
    Limits l;
    l.yes = -1.f;
    l.no = INFINITY;
    if (!(alpha > 1e-20f) || !(t < 1e18f)) return l;   // (alpha 0: every test in FP32)
    const float a = (t * 0.9998f - err) * inv_scale, b = (t * 1.0002f + err) * inv_scale;
    if (a > 0.f) l.yes = a * a * 0.99999f;
    l.no = b * b * 1.00001f + 1.f;
    return l;
}

__device__ __forceinline__ void cp_async16(uint32_t *dst, const uint8_t *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                     static_cast<uint32_t>(__cvta_generic_to_shared(dst))),
                 "l"(src)
                 : "memory");
}

// The FP32 prune distances of the owner to this lane's two rows, the chain of
// prune_dist.  The rows pass through s.rows a quarter at a time (a quarter is as long as
// a code row): copied by consecutive lanes, read back a row a lane.  Loaded a row a
// lane straight from global memory, each 16-byte load of a warp touched 32 lines, and
// the L1 pipe was the kernel's limit (100k DEEP-like owners 1.41 ms, now 1.16).
template <int W, class Pool>
__device__ __forceinline__ void owner_dists(Pool &s, int nr, bool two, float &d0, float &d1) {
    constexpr int kStride = Pool::kStride, kVec = W / 4;
    const int lane = threadIdx.x & 31;
    f2_t a0 = 0ull, a1 = 0ull;
#pragma unroll 1
    for (int c = 0; c < 4; ++c) {
        for (int u = lane; u < nr * kVec; u += 32) {
            const int r = u / kVec, f = u - r * kVec;
            const float *x = s.rptr[r];
            if (x) cp_async16(s.rows + r * kStride + 4 * f, reinterpret_cast<const uint8_t *>(x + c * W + 4 * f));
        }
        asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
        __syncwarp();
        const ulonglong2 *v = reinterpret_cast<const ulonglong2 *>(s.vrow + c * kVec);
        const ulonglong2 *x0 = reinterpret_cast<const ulonglong2 *>(s.rows + lane * kStride);
        const ulonglong2 *x1 = reinterpret_cast<const ulonglong2 *>(s.rows + (lane + 32) * kStride);
#pragma unroll
        for (int f = 0; f < kVec; ++f) {
            const ulonglong2 o = v[f];
            a0 = chain2(a0, o, x0[f], 0);
            if (two) a1 = chain2(a1, o, x1[f], 0);
        }
        __syncwarp();
    }
    d0 = chain2_final(a0, 0);
    if (two) d1 = chain2_final(a1, 0);
}

template <int W, bool kExact>
__global__ void __launch_bounds__(kCodeWarps * 32, code_blocks<W, kExact>())
    prune_code_kernel(const __grid_constant__ PruneArgs a, int chunk) {
    using Pool = CodePool<W, kExact>;
    constexpr int kStride = Pool::kStride, kVec = W / 4;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    Pool &s = reinterpret_cast<Pool *>(smem_raw)[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    const int R = a.R;
    float inv_scale = 0.f, err = 0.f;
    if (!kExact) {
        inv_scale = a.code_params->inv_scale;
        err = a.code_params->err;
    }
    for (;;) {
        int32_t claim = 0;
        if (lane == 0) claim = atomicAdd(a.work, chunk);
        const int64_t i0 = __shfl_sync(0xffffffffu, claim, 0);
        if (i0 >= a.n_owners) break;
        const int64_t i1 = min(a.n_owners, i0 + chunk);
        for (int64_t i = i0; i < i1; ++i) {
            const int32_t owner = a.owner_ids ? a.owner_ids[i] : (int32_t)(a.owner_base + i);
            int64_t c_lo = 0, c_hi = 0;
            if (a.csr_offs) {
                c_lo = a.csr_offs[i];
                c_hi = a.csr_offs[i + 1];
            }
            if (a.skip_empty_csr && c_hi == c_lo) continue;
            const int64_t nr_raw = (int64_t)a.lenA + a.lenB + (c_hi - c_lo);
            if (nr_raw > kPool) {
                if (lane == 0) a.ovf_list[atomicAdd(a.ovf_count, 1ull)] = (int32_t)i;
                continue;
            }
            const int nr = (int)nr_raw;
            // 1. the pool's ids, and every row (and the owner's) on its way
            int32_t id[2];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int j = lane + 32 * h;
                int32_t c = -1;
                if (j < nr) {
                    if (j < a.lenA) {
                        c = a.listA[(int64_t)owner * a.lenA + j];
                    } else if (j < a.lenA + a.lenB) {
                        c = a.listB[i * a.strideB + (j - a.lenA)];
                        if (c >= 0) c += a.offB;
                    } else {
                        c = a.csr_ids[c_lo + (j - a.lenA - a.lenB)];
                    }
                    if (c == owner) c = -1;
                }
                id[h] = c;
                s.id[j] = c;
                if (!kExact) s.rptr[j] = c >= 0 ? seg_row(a.segs, c, 4 * W) : nullptr;
            }
            const bool two = nr > 32;
            float e0 = INFINITY, e1 = INFINITY;   // filter: FP32 distances to the owner
            if (!kExact) {   // the order is that of the FP32 chain
                const float *orow = seg_row(a.segs, owner, 4 * W);
                if (lane < W) s.vrow[lane] = ldg4(orow + 4 * lane);
                __syncwarp();
                owner_dists<W>(s, nr, two, e0, e1);
            }
            __syncwarp();
            if (kExact && lane < kVec) cp_async16(s.owner + 4 * lane, a.codes + (int64_t)owner * (4 * W) + 16 * lane);
            for (int c = lane; c < nr * kVec; c += 32) {
                const int r = c / kVec, f = c - r * kVec;
                const int32_t g = s.id[r];
                if (g >= 0) cp_async16(s.rows + r * kStride + 4 * f, a.codes + (int64_t)g * (4 * W) + 16 * f);
            }
            asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;" ::: "memory");
            __syncwarp();
            // 2. keys: distance to the owner, id, slot (none repeats)
            uint32_t nv = 0u, n0 = 0u, n1 = 0u, v0 = 0u, v1 = 0u;
            const uint4 *r0 = reinterpret_cast<const uint4 *>(s.rows + lane * kStride);
            const uint4 *r1 = reinterpret_cast<const uint4 *>(s.rows + (lane + 32) * kStride);
#pragma unroll
            for (int f = 0; f < kVec; ++f) {
                uint4 o = make_uint4(0u, 0u, 0u, 0u);
                if (kExact) {
                    o = reinterpret_cast<const uint4 *>(s.owner)[f];
                    nv = __dp4a(o.x, o.x, __dp4a(o.y, o.y, __dp4a(o.z, o.z, __dp4a(o.w, o.w, nv))));
                }
                const uint4 x = r0[f];
                n0 = __dp4a(x.x, x.x, __dp4a(x.y, x.y, __dp4a(x.z, x.z, __dp4a(x.w, x.w, n0))));
                if (kExact) v0 = __dp4a(x.x, o.x, __dp4a(x.y, o.y, __dp4a(x.z, o.z, __dp4a(x.w, o.w, v0))));
                if (two) {
                    const uint4 y = r1[f];
                    n1 = __dp4a(y.x, y.x, __dp4a(y.y, y.y, __dp4a(y.z, y.z, __dp4a(y.w, y.w, n1))));
                    if (kExact) v1 = __dp4a(y.x, o.x, __dp4a(y.y, o.y, __dp4a(y.z, o.z, __dp4a(y.w, o.w, v1))));
                }
            }
            s.norm[lane] = (int32_t)n0;
            s.norm[lane + 32] = (int32_t)n1;
            unsigned long long K[2];
            if (!kExact) {   // (repeats share a key: one position, the next one empty)
                K[0] = id[0] >= 0 ? ((unsigned long long)__float_as_uint(e0) << 32) | (uint32_t)id[0] : ~0ull;
                K[1] = id[1] >= 0 ? ((unsigned long long)__float_as_uint(e1) << 32) | (uint32_t)id[1] : ~0ull;
                s.order[lane] = ~0ull;
                s.order[lane + 32] = ~0ull;
            } else {
                K[0] = (id[0] >= 0 ? ((unsigned long long)(nv + n0 - 2u * v0) << 37) | ((unsigned long long)(uint32_t)id[0] << 6)
                                   : ~63ull) | (unsigned)lane;
                K[1] = (id[1] >= 0 ? ((unsigned long long)(nv + n1 - 2u * v1) << 37) | ((unsigned long long)(uint32_t)id[1] << 6)
                                   : ~63ull) | (unsigned)(lane + 32);
            }
            s.key[lane] = K[0];
            s.key[lane + 32] = K[1];
            __syncwarp();
            // 3. position = number of smaller keys
            {
                int p0 = 0, p1 = 0;
                const ulonglong2 *kk = reinterpret_cast<const ulonglong2 *>(s.key);
                const int half = two ? 32 : 16;
#pragma unroll 8
                for (int k = 0; k < half; ++k) {
                    const ulonglong2 q = kk[k];
                    p0 += (q.x < K[0] ? 1 : 0) + (q.y < K[0] ? 1 : 0);
                    p1 += (q.x < K[1] ? 1 : 0) + (q.y < K[1] ? 1 : 0);
                }
                if (!kExact) {
                    if (id[0] >= 0) {
                        s.order[p0] = K[0];
                        s.slot[p0] = lane;
                    }
                    if (id[1] >= 0) {
                        s.order[p1] = K[1];
                        s.slot[p1] = lane + 32;
                    }
                } else {
                    s.order[p0] = K[0];
                    if (two) s.order[p1] = K[1];
                    else s.order[lane + 32] = K[1];
                }
            }
            __syncwarp();
            K[0] = s.order[lane];
            K[1] = s.order[lane + 32];
            bool live0, live1;   // live positions: valid and not a repeat of the previous id
            if (kExact) {
                id[0] = (int32_t)((K[0] >> 6) & 0x7fffffffull);
                id[1] = (int32_t)((K[1] >> 6) & 0x7fffffffull);
                const int32_t pr0 = lane ? (int32_t)((s.order[lane - 1] >> 6) & 0x7fffffffull) : -1;
                const int32_t pr1 = (int32_t)((s.order[lane + 31] >> 6) & 0x7fffffffull);
                live0 = K[0] < ~63ull && pr0 != id[0];
                live1 = K[1] < ~63ull && pr1 != id[1];
            } else {
                id[0] = (int32_t)(uint32_t)K[0];
                id[1] = (int32_t)(uint32_t)K[1];
                live0 = K[0] != ~0ull;
                live1 = K[1] != ~0ull;
            }
            const unsigned long long live = (unsigned long long)__ballot_sync(0xffffffffu, live0) |
                                            ((unsigned long long)__ballot_sync(0xffffffffu, live1) << 32);
            unsigned long long kept = 0ull;
            if (a.keep_all_if_fit && __popcll(live) <= R) {
                kept = live;
            } else {
                // 4. the walk
                uint32_t x0[W], x1[W];
                const int s0 = kExact ? (int)(K[0] & 63ull) : live0 ? s.slot[lane] : 0;
                const int s1 = kExact ? (int)(K[1] & 63ull) : live1 ? s.slot[lane + 32] : 0;
                const uint4 *q0 = reinterpret_cast<const uint4 *>(s.rows + s0 * kStride);
                const uint4 *q1 = reinterpret_cast<const uint4 *>(s.rows + s1 * kStride);
#pragma unroll
                for (int f = 0; f < kVec; ++f) {
                    const uint4 x = q0[f];
                    x0[4 * f] = x.x;
                    x0[4 * f + 1] = x.y;
                    x0[4 * f + 2] = x.z;
                    x0[4 * f + 3] = x.w;
                    const uint4 y = q1[f];
                    x1[4 * f] = y.x;
                    x1[4 * f + 1] = y.y;
                    x1[4 * f + 2] = y.z;
                    x1[4 * f + 3] = y.w;
                }
                const int32_t m0 = s.norm[s0], m1 = s.norm[s1];
                const float dv0 = kExact ? (float)(uint32_t)(K[0] >> 37) : __uint_as_float((uint32_t)(K[0] >> 32));
                const float dv1 = kExact ? (float)(uint32_t)(K[1] >> 37) : __uint_as_float((uint32_t)(K[1] >> 32));
                const Limits l0 = kExact ? Limits() : limits_of(dv0, a.alpha, err, inv_scale);
                const Limits l1 = kExact ? Limits() : limits_of(dv1, a.alpha, err, inv_scale);
                // does the kept row, at code distance S, occlude this lane's position?
                auto occludes = [&](int32_t S, float dv, const Limits &l, bool is_open, int32_t mine, int p) -> bool {
                    const float f = (float)S;
                    if (kExact) return fmaf(a.alpha, f, -dv) <= 0.f;
                    bool r = f <= l.yes;
                    if (!r && f <= l.no && is_open) {   // left open by the codes: the FP32 distance
                        r = fmaf(a.alpha, far_dist<W>(a.segs, (int32_t)(uint32_t)s.order[p], mine), -dv) <= 0.f;
                    }
                    return r;
                };
                unsigned long long open = live;
                int nk = 0;
                while (open && nk < R) {
                    const int p = __ffsll((long long)open) - 1;
                    kept |= 1ull << p;
                    ++nk;
                    open &= open - 1ull;
                    if (!open) break;
                    const int ss = kExact ? (int)(reinterpret_cast<const uint32_t *>(s.order)[2 * p] & 63u) : s.slot[p];
                    const uint4 *row = reinterpret_cast<const uint4 *>(s.rows + ss * kStride);
                    const int32_t ns = s.norm[ss];
                    unsigned d0 = 0u, d1 = 0u;
                    const unsigned o0 = (unsigned)open, o1 = (unsigned)(open >> 32);
                    const bool m_open0 = (o0 >> lane) & 1u, m_open1 = (o1 >> lane) & 1u;
                    // (a half without open positions is left out)
                    if (o0 && o1) {
                        uint32_t t0 = 0u, t1 = 0u;
#pragma unroll
                        for (int f = 0; f < kVec; ++f) {
                            const uint4 o = row[f];
                            t0 = __dp4a(x0[4 * f], o.x, __dp4a(x0[4 * f + 1], o.y, __dp4a(x0[4 * f + 2], o.z, __dp4a(x0[4 * f + 3], o.w, t0))));
                            t1 = __dp4a(x1[4 * f], o.x, __dp4a(x1[4 * f + 1], o.y, __dp4a(x1[4 * f + 2], o.z, __dp4a(x1[4 * f + 3], o.w, t1))));
                        }
                        d0 = __ballot_sync(0xffffffffu, occludes(ns + m0 - 2 * (int32_t)t0, dv0, l0, m_open0, id[0], p));
                        d1 = __ballot_sync(0xffffffffu, occludes(ns + m1 - 2 * (int32_t)t1, dv1, l1, m_open1, id[1], p));
                    } else {
                        uint32_t t0 = 0u, t1 = 0u;
                        if (o0) {
#pragma unroll
                            for (int f = 0; f < kVec; ++f) {
                                const uint4 o = row[f];
                                t0 = __dp4a(x0[4 * f], o.x, __dp4a(x0[4 * f + 1], o.y, t0));
                                t1 = __dp4a(x0[4 * f + 2], o.z, __dp4a(x0[4 * f + 3], o.w, t1));
                            }
                            d0 = __ballot_sync(0xffffffffu, occludes(ns + m0 - 2 * (int32_t)(t0 + t1), dv0, l0, m_open0, id[0], p));
                        } else {
#pragma unroll
                            for (int f = 0; f < kVec; ++f) {
                                const uint4 o = row[f];
                                t0 = __dp4a(x1[4 * f], o.x, __dp4a(x1[4 * f + 1], o.y, t0));
                                t1 = __dp4a(x1[4 * f + 2], o.z, __dp4a(x1[4 * f + 3], o.w, t1));
                            }
                            d1 = __ballot_sync(0xffffffffu, occludes(ns + m1 - 2 * (int32_t)(t0 + t1), dv1, l1, m_open1, id[1], p));
                        }
                    }
                    open &= ~((unsigned long long)d0 | ((unsigned long long)d1 << 32));
                }
            }
            // 5. output in (distance, id) order: the kept positions
            {
                const int nk = __popcll(kept);
                int32_t *out = a.out + (a.out_by_index ? i : (int64_t)owner) * R;
                const bool k0 = (kept >> lane) & 1ull, k1 = (kept >> (lane + 32)) & 1ull;
                if (k0) out[__popcll(kept & ((1ull << lane) - 1ull))] = id[0];
                if (k1) out[__popcll(kept & ((1ull << (lane + 32)) - 1ull))] = id[1];
                for (int j = nk + lane; j < R; j += 32) out[j] = -1;
                if (a.eu) {
                    const bool e0 = k0 && id[0] >= a.emit_lo && id[0] < a.emit_hi;
                    const bool e1 = k1 && id[1] >= a.emit_lo && id[1] < a.emit_hi;
                    const unsigned b0 = __ballot_sync(0xffffffffu, e0);
                    const unsigned b1 = __ballot_sync(0xffffffffu, e1);
                    const int cnt = __popc(b0) + __popc(b1);
                    int base = 0;
                    if (lane == 0 && cnt) base = (int)atomicAdd(a.ecount, (unsigned long long)cnt);
                    base = __shfl_sync(0xffffffffu, base, 0);
                    if (e0) {
                        const int slot = base + __popc(b0 & lanemask_lt());
                        a.eu[slot] = id[0];
                        a.ev[slot] = owner;
                    }
                    if (e1) {
                        const int slot = base + __popc(b0) + __popc(b1 & lanemask_lt());
                        a.eu[slot] = id[1];
                        a.ev[slot] = owner;
                    }
                }
            }
            __syncwarp();   // the owner's shared state is free
        }
    }
}

template <int W, bool kExact>
cudaError_t launch_code_t(const PruneArgs &a, cudaStream_t st) {
    auto kern = prune_code_kernel<W, kExact>;
    constexpr int smem = kCodeWarps * (int)sizeof(CodePool<W, kExact>);
    static GridCache cache;
    int64_t grid = 0;
    cudaError_t e = cached_grid(cache, grid, [&](int dev, int &blocks) {
        cudaError_t r = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (r != cudaSuccess) return r;
        cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
        int sms = 0, per_sm = 0;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        r = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kCodeWarps * 32, smem);
        blocks = sms * (per_sm < 1 ? 1 : per_sm);
        return r;
    });
    if (e != cudaSuccess) return e;
    const int chunk = a.skip_empty_csr ? 8 : 2;
    const int64_t want = (a.n_owners + (int64_t)kCodeWarps * chunk - 1) / ((int64_t)kCodeWarps * chunk);
    if (want < grid) grid = want;
    kern<<<(unsigned)grid, kCodeWarps * 32, smem, st>>>(a, chunk);
    note_launches(1);
    return cudaGetLastError();
}

}  // namespace

bool prune_code_ok(int dim, int metric) { return metric == 0 && (dim == 64 || dim == 96 || dim == 128); }

cudaError_t launch_prune_code(const PruneArgs &a, cudaStream_t st) {
    if (!a.codes || !prune_code_ok(a.dim, a.metric)) return cudaErrorInvalidValue;
    if (a.code_params)
        return a.dim == 64   ? launch_code_t<16, false>(a, st)
               : a.dim == 96 ? launch_code_t<24, false>(a, st)
                             : launch_code_t<32, false>(a, st);
    return a.dim == 64   ? launch_code_t<16, true>(a, st)
           : a.dim == 96 ? launch_code_t<24, true>(a, st)
                         : launch_code_t<32, true>(a, st);
}

}  // namespace rnsm
