// rows.cu -- the kernels around gemm.cu of a pass over many token rows (prompt processing).
//
// The persistent pass kernel (pass_kernel.cu) is built for the few rows of a decoding pass, where a
// layer is a chain of short dependent steps.  With hundreds of rows a layer is matrix products
// and attention that fill the GPU by themselves, so each step is its own kernel here:
//     k_rows_embed   token embedding, first RMSNorm
//     gemm.cu        q|k|v                              -> qkv
//     k_rows_rope    QK-norm, RoPE, paged K/V write     -> q, cache
//     k_rows_attn    causal attention over the cache    -> attn
//     gemm.cu        o                                  -> y
//     k_rows_norm    residual add, RMSNorm              -> h, x
//     gemm.cu        gate|up with SiLU(gate) * up       -> act
//     gemm.cu        down                               -> y
//     k_rows_norm    residual add, next layer's RMSNorm -> h, x
//     k_rows_final   final RMSNorm of the read-out rows
//
// Every value is computed with the pass kernel's arithmetic, operation for operation (K slices and
// their order, key partition of the attention, order of every sum, every rounding to bf16), so the
// cached K/V and the logits of a prompt equal, bit for bit, those of decoding the same tokens.
#include <algorithm>

#include "attn.cuh"
#include "common.cuh"
#include "pbd_internal.h"

namespace pbd {

constexpr int RW_THREADS = 256;  // one warp per row (or row and tile), eight a block

// segment of row m, and its sequence position
__device__ __forceinline__ int row_seg(const RowsArgs &a, int m) {
    int s = 0;
    while (s + 1 < a.n_seg && m >= a.segs[s + 1].row0) ++s;
    return s;
}

// 1/sqrt(mean + eps) from a row's sum of squares, as row_rms in pass_kernel.cu
__device__ __forceinline__ float rms_scale(float sum, int H, float eps) {
    return __fdiv_rn(1.0f, __fsqrt_rn(__fadd_rn(__fdiv_rn(sum, (float)H), eps)));
}

__device__ __forceinline__ float warp_sum_butterfly(float s) {
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) s = __fadd_rn(s, __shfl_xor_sync(0xffffffffu, s, off));
    return s;
}

// four bf16 of a row times its scale and gain: bf16(g * bf16(h * rs))
__device__ __forceinline__ uint2 norm4(uint2 h, uint2 g, float rs) {
    uint2 o;
    const uint32_t hw[2] = {h.x, h.y}, gw[2] = {g.x, g.y};
    uint32_t ow[2];
#pragma unroll
    for (int e = 0; e < 2; ++e) {
        const float2 f = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&hw[e]));
        const __nv_bfloat162 r = __hmul2(*reinterpret_cast<const __nv_bfloat162 *>(&gw[e]),
                                         __floats2bfloat162_rn(__fmul_rn(f.x, rs), __fmul_rn(f.y, rs)));
        ow[e] = *reinterpret_cast<const uint32_t *>(&r);
    }
    o.x = ow[0];
    o.y = ow[1];
    return o;
}

// ids[m] -> h[m] and x[m] = RMSNorm of it with the first layer's gain.  An id outside [0, V) latches
// DEV_BAD_TOKEN and reads row 0.
__global__ void __launch_bounds__(RW_THREADS) k_rows_embed(const __grid_constant__ RowsArgs a, const int *ids,
                                                           const bf16 *__restrict__ embed_tiled,
                                                           const bf16 *__restrict__ gain) {
    const int lane = threadIdx.x & 31, H = a.dm.H, nt = H / TILE_ROWS;
    pdl_begin();
    for (int m = blockIdx.x * (RW_THREADS / 32) + (threadIdx.x >> 5); m < a.M; m += gridDim.x * (RW_THREADS / 32)) {
        int tok = ids[m];
        if (tok < 0 || tok >= a.dm.V) {
            if (lane == 0) latch_error(a.status, DEV_BAD_TOKEN);
            tok = 0;
        }
        float sum = 0.f;
        for (int t = 0; t < nt; ++t) {
            // lane l adds elements l, l + 32, l + 64, l + 96 of the tile in that order, then a butterfly
            float s = 0.f;
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const int f = t * TILE_ROWS + lane + 32 * e;
                const bf16 v = *tiled_at(embed_tiled, H, tok, f);
                a.h[(size_t)m * H + f] = v;
                const float w = bf2f(v);
                s = e == 0 ? __fmul_rn(w, w) : __fadd_rn(s, __fmul_rn(w, w));
            }
            s = warp_sum_butterfly(s);
            sum = t == 0 ? s : __fadd_rn(sum, s);
        }
        const float rs = rms_scale(sum, H, a.dm.eps);
        __syncwarp();
        for (int t = 0; t < nt; ++t) {
            const int f = t * TILE_ROWS + 4 * lane;
            const uint2 hv = *reinterpret_cast<const uint2 *>(a.h + (size_t)m * H + f);
            *reinterpret_cast<uint2 *>(a.x + (size_t)m * H + f) =
                norm4(hv, *reinterpret_cast<const uint2 *>(gain + f), rs);
        }
    }
}

// h[m] += y[m] (both already rounded to bf16, the sum too), x[m] = RMSNorm of it with `gain` (not
// when gain is null).  The sum of squares of a 128-feature tile adds lane l's features 4l..4l+3 in
// order, then a butterfly; tiles in order.  Bound by L2 and HBM: 8 bytes a feature.
__global__ void __launch_bounds__(RW_THREADS) k_rows_norm(const __grid_constant__ RowsArgs a,
                                                          const bf16 *__restrict__ gain) {
    constexpr int NT = 8;  // tiles kept in registers (H <= 1024; longer rows are read again)
    const int lane = threadIdx.x & 31, H = a.dm.H, nt = H / TILE_ROWS;
    pdl_begin();
    for (int m = blockIdx.x * (RW_THREADS / 32) + (threadIdx.x >> 5); m < a.M; m += gridDim.x * (RW_THREADS / 32)) {
        uint2 *hp = reinterpret_cast<uint2 *>(a.h + (size_t)m * H) + lane;
        const uint2 *yp = reinterpret_cast<const uint2 *>(a.y + (size_t)m * H) + lane;
        uint2 keep[NT];
        float sum = 0.f;
        for (int t0 = 0; t0 < nt; t0 += NT) {
            uint2 hv[NT], yv[NT];
#pragma unroll
            for (int u = 0; u < NT; ++u)
                if (t0 + u < nt) hv[u] = hp[(t0 + u) * 32], yv[u] = yp[(t0 + u) * 32];
#pragma unroll
            for (int u = 0; u < NT; ++u) {
                if (t0 + u >= nt) break;
                const __nv_bfloat162 *h2 = reinterpret_cast<const __nv_bfloat162 *>(&hv[u]);
                const __nv_bfloat162 *y2 = reinterpret_cast<const __nv_bfloat162 *>(&yv[u]);
                const float2 ha = __bfloat1622float2(h2[0]), hb = __bfloat1622float2(h2[1]);
                const float2 ya = __bfloat1622float2(y2[0]), yb = __bfloat1622float2(y2[1]);
                const float v[4] = {rbf(__fadd_rn(ha.x, ya.x)), rbf(__fadd_rn(ha.y, ya.y)), rbf(__fadd_rn(hb.x, yb.x)),
                                    rbf(__fadd_rn(hb.y, yb.y))};
                keep[u] = make_uint2(pack_bf162(v[0], v[1]), pack_bf162(v[2], v[3]));
                hp[(t0 + u) * 32] = keep[u];
                float s = __fmul_rn(v[0], v[0]);
#pragma unroll
                for (int e = 1; e < 4; ++e) s = __fadd_rn(s, __fmul_rn(v[e], v[e]));
                s = warp_sum_butterfly(s);
                sum = t0 + u == 0 ? s : __fadd_rn(sum, s);
            }
        }
        if (gain == nullptr) continue;
        const float rs = rms_scale(sum, H, a.dm.eps);
        const uint2 *gp = reinterpret_cast<const uint2 *>(gain) + lane;
        uint2 *xp = reinterpret_cast<uint2 *>(a.x + (size_t)m * H) + lane;
        if (nt <= NT) {
#pragma unroll
            for (int u = 0; u < NT; ++u)
                if (u < nt) xp[u * 32] = norm4(keep[u], __ldg(gp + u * 32), rs);
        } else {
            for (int t = 0; t < nt; ++t) xp[t * 32] = norm4(hp[t * 32], __ldg(gp + t * 32), rs);
        }
    }
}

// q|k|v of one row: per-head RMSNorm and RoPE of q and k; q to its buffer, k and v to the cache
// pages.  A block per row, a warp per 128-feature tile (every eighth one): lane l holds features
// 4l..4l+3, as in reduce_qkv (pass_kernel.cu).  Bound by L2: 8 bytes a feature, read and written.
template <int DH>
__global__ void __launch_bounds__(RW_THREADS) k_rows_rope(const __grid_constant__ RowsArgs a, int layer,
                                                          const bf16 *__restrict__ q_norm,
                                                          const bf16 *__restrict__ k_norm,
                                                          const float2 *__restrict__ rope_cs) {
    constexpr int LPH = DH / 4;  // lanes per head
    constexpr int U = 4;         // tiles whose loads go out together
    const Dims &dm = a.dm;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int qw = dm.Hq * DH, kvw = dm.Hkv * DH, nq = (qw + 2 * kvw) / TILE_ROWS;
    const int hl = lane / LPH, e0 = 4 * (lane % LPH);
    const bool lo = e0 < DH / 2;
    auto gain4 = [&](const bf16 *g, float (&o)[4]) {
        const uint2 raw = __ldg(reinterpret_cast<const uint2 *>(g + (size_t)layer * DH + e0));
        const float2 p = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&raw.x));
        const float2 q = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&raw.y));
        o[0] = p.x, o[1] = p.y, o[2] = q.x, o[3] = q.y;
    };
    float gq[4], gk[4];
    gain4(q_norm, gq);
    gain4(k_norm, gk);
    pdl_begin();
    for (int m = blockIdx.x; m < a.M; m += gridDim.x) {
        const RowSeg sg = a.segs[row_seg(a, m)];
        const int pos = sg.pos0 + m - sg.row0;
        const float4 *c4 = reinterpret_cast<const float4 *>(rope_cs + (size_t)pos * (DH / 2) + (e0 % (DH / 2)));
        const float4 ca = __ldg(c4), cb = __ldg(c4 + 1);
        const float cs[4] = {ca.x, ca.z, cb.x, cb.z}, sn[4] = {ca.y, ca.w, cb.y, cb.w};
        const size_t slot = ((size_t)layer * a.kv.n_pages + a.kv.page_table[sg.seq * a.kv.pages_per_seq + pos / PAGE]) * dm.Hkv;
        for (int t0 = warp; t0 < nq; t0 += U * (RW_THREADS / 32)) {
            uint2 raw[U];
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int ft = (t0 + u * (RW_THREADS / 32)) * TILE_ROWS;
                if (ft < qw + 2 * kvw) raw[u] = *reinterpret_cast<const uint2 *>(a.qkv + (size_t)m * (qw + 2 * kvw) + ft + 4 * lane);
            }
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int ft = (t0 + u * (RW_THREADS / 32)) * TILE_ROWS;
                if (ft >= qw + 2 * kvw) break;  // (uniform)
                const int kind = ft < qw ? 0 : (ft < qw + kvw ? 1 : 2);
                const int head = (ft - (kind == 0 ? 0 : (kind == 1 ? qw : qw + kvw))) / DH + hl;
                uint2 out = raw[u];
                if (kind < 2) {
                    const float2 ya = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&raw[u].x));
                    const float2 yb = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&raw[u].y));
                    float y[4] = {ya.x, ya.y, yb.x, yb.y};
                    float ss = __fmul_rn(y[0], y[0]);
#pragma unroll
                    for (int j = 1; j < 4; ++j) ss = __fadd_rn(ss, __fmul_rn(y[j], y[j]));
#pragma unroll
                    for (int off = LPH / 2; off >= 1; off >>= 1) ss = __fadd_rn(ss, __shfl_xor_sync(0xffffffffu, ss, off));
                    const float rs = rms_scale(ss, DH, dm.eps);
                    float z[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) y[j] = rbf(__fmul_rn(kind == 0 ? gq[j] : gk[j], rbf(__fmul_rn(y[j], rs))));
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float partner = __shfl_xor_sync(0xffffffffu, y[j], LPH / 2);
                        z[j] = lo ? __fsub_rn(__fmul_rn(y[j], cs[j]), __fmul_rn(partner, sn[j]))
                                  : __fadd_rn(__fmul_rn(y[j], cs[j]), __fmul_rn(partner, sn[j]));
                    }
                    out = make_uint2(pack_bf162(z[0], z[1]), pack_bf162(z[2], z[3]));
                }
                bf16 *dst = kind == 0 ? a.q + ((size_t)m * dm.Hq + head) * DH + e0
                                      : static_cast<bf16 *>(kind == 1 ? a.kv.k : a.kv.v) +
                                            ((slot + head) * PAGE + (pos % PAGE)) * DH + e0;
                *reinterpret_cast<uint2 *>(dst) = out;
            }
        }
    }
}

// ------------------------------------------------------------------ attention
//
// One CTA: 128 (row, head) pairs of one sequence's segment and KV head, 16 per compute warp, against
// the cached keys up to the last row's position, in the pass kernel's partition: 128-key splits, each
// one or two partial results of HALF keys computed in 32-key chunks with a running maximum, combined
// in key order relative to the row's overall maximum.  The pass kernel stores the partial
// results and merges them afterwards; here a first sweep over the keys finds the overall maximum
// (scores only), and the second sweep computes each partial result and adds it to the row's sums
// at once, in registers.  One more QK^T per key replaces 520 bytes of partial results written
// and read back per (row, head, partial).
//
// Warp 8 streams units of 128 keys of K (first sweep) or K, then V (second) into a ring: one tiled
// TMA per 16-token page and 64-dim half.
//
// Bound: latency of legacy mma.sync in two warps per SM quarter (4096 rows: 352 us a layer; 497 us with
// the scores' MMAs in one chain after another and swizzled addresses computed per fragment; 387 us
// as two CTAs of four warps).  The tcgen05 tensor core is not used because its summation order
// differs from the decoding pass's.
constexpr int RA_WARPS = 8;
constexpr int RA_THREADS = 32 * RA_WARPS + 128;  // the producer's warpgroup has one warp with work
constexpr int RA_UNITS = 4;

template <int DH>
struct RaLayout {
    static constexpr int SUB = ATT_SPLIT * 128;  // 128 keys x 64 dims, 128-byte swizzle
    static constexpr int UNIT = (DH / 64) * SUB;
    static constexpr int TOTAL = RA_UNITS * UNIT + 1024;
};

template <int DH>
__global__ void __launch_bounds__(RA_THREADS, 1)
    k_rows_attn(const __grid_constant__ CUtensorMap kmap, const __grid_constant__ CUtensorMap vmap,
                const __grid_constant__ RowsArgs a, int layer, const RowsAttn *__restrict__ work, int n_work) {
    using LY = RaLayout<DH>;
    constexpr int KS = DH / 16, DT = DH / 8, SUBS = DH / 64;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *ring = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ uint64_t full[RA_UNITS], empty[RA_UNITS];
    __shared__ int s_abort;
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const Dims &dm = a.dm;
    const int grp = dm.Hq / dm.Hkv;
    if (threadIdx.x == 0) {
        for (int i = 0; i < RA_UNITS; ++i) {
            mbar_init(&full[i], 1);
            mbar_init(&empty[i], RA_WARPS);
        }
        s_abort = 0;
        fence_mbarrier_init();
        prefetch_tensormap(&kmap);
        prefetch_tensormap(&vmap);
    }
    __syncthreads();
    pdl_begin();
    int slot = 0;
    // registers: the producer's warpgroup gives up 128 x 128 of the launch's 3 x 128 x 168, the two
    // compute warpgroups take 128 x 56 each
    if (warp >= RA_WARPS) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
        if (warp > RA_WARPS) return;
        // ---- producer warp: a lane per page and half
        uint32_t ph = 1;
        int issued = 0;
        bool ok = true;
        // this pass's own K/V were written by generic stores of an earlier kernel
        fence_proxy_async_global();
        for (int w = blockIdx.x; ok && w < n_work; w += gridDim.x) {
            const RowsAttn wk = work[w];
            const RowSeg sg = a.segs[wk.seg];
            const int last = sg.pos0 + min(sg.n - 1, (wk.q0 + 16 * RA_WARPS - 1) / grp);  // last visible key
            const int ns = last / ATT_SPLIT + 1;
            for (int u = 0; u < 3 * ns; ++u) {  // K of every split, then K and V of every split
                const int s = u < ns ? u : (u - ns) >> 1;
                const bool v = u >= ns && ((u - ns) & 1);
                if (!mbar_wait(&empty[slot], ph, a.status, DEV_TIMEOUT_SLOT, &s_abort)) {
                    ok = false;
                    break;
                }
                const int npg = min(ATT_SPLIT / PAGE, last / PAGE - s * (ATT_SPLIT / PAGE) + 1);
                if (lane == 0) mbar_arrive_expect_tx(&full[slot], (uint32_t)(npg * SUBS * PAGE * 128));
                __syncwarp();
                if (lane < npg * SUBS) {
                    const int p = lane / SUBS, sub = lane % SUBS;
                    const int page = a.kv.page_table[sg.seq * a.kv.pages_per_seq + s * (ATT_SPLIT / PAGE) + p];
                    tma_load_2d(ring + (size_t)slot * LY::UNIT + sub * LY::SUB + p * PAGE * 128, v ? &vmap : &kmap, sub * 64,
                                ((layer * a.kv.n_pages + page) * dm.Hkv + wk.g) * PAGE, &full[slot]);
                }
                ++issued;
                if (++slot == RA_UNITS) slot = 0, ph ^= 1;
            }
        }
        if (*(volatile int *)&s_abort)  // error path: the copies in flight get a bounded chance to land
            for (int h = issued > RA_UNITS ? issued - RA_UNITS : 0; h < issued; ++h)
                mbar_wait(&full[h % RA_UNITS], (h / RA_UNITS) & 1, nullptr, 0, nullptr);
        return;
    }
    // ---- compute warps
    asm volatile("setmaxnreg.inc.sync.aligned.u32 224;");
    const int gq = lane >> 2, tq = lane & 3;
    const float scale = a.att_scale;
    const int HALF = ATT_SPLIT / a.att_subs;
    const uint32_t koff = attn_k_lane(lane), voff = attn_v_lane(lane);
    uint32_t ph = 0;
    for (int w = blockIdx.x; w < n_work; w += gridDim.x) {
        const RowsAttn wk = work[w];
        const RowSeg sg = a.segs[wk.seg];
        const int last = sg.pos0 + min(sg.n - 1, (wk.q0 + 16 * RA_WARPS - 1) / grp);
        const int ns = last / ATT_SPLIT + 1, T = sg.pos0 + sg.n, QV = sg.n * grp;
        const int qv0 = wk.q0 + warp * 16 + gq, qv1 = qv0 + 8;
        const bool val0 = qv0 < QV, val1 = qv1 < QV;
        const int i0 = val0 ? qv0 / grp : 0, i1 = val1 ? qv1 / grp : 0;
        const int h0 = wk.g * grp + (val0 ? qv0 % grp : 0), h1 = wk.g * grp + (val1 ? qv1 % grp : 0);
        const int lim0 = val0 ? sg.pos0 + i0 : -1, lim1 = val1 ? sg.pos0 + i1 : -1;  // last visible keys
        // the warp's last visible key (-1: no rows), and the last key that all its rows see
        const int wq0 = wk.q0 + warp * 16;
        const int wlast = wq0 < QV ? sg.pos0 + min(sg.n - 1, (wq0 + 15) / grp) : -1;
        const int wall = wq0 + 15 < QV ? sg.pos0 + wq0 / grp : -1;
        uint32_t qa[KS][4];
        {
            const bf16 *q0 = a.q + ((size_t)(sg.row0 + i0) * dm.Hq + h0) * DH + 2 * tq;
            const bf16 *q1 = a.q + ((size_t)(sg.row0 + i1) * dm.Hq + h1) * DH + 2 * tq;
#pragma unroll
            for (int ks = 0; ks < KS; ++ks) {
                qa[ks][0] = val0 ? *reinterpret_cast<const unsigned *>(q0 + ks * 16) : 0u;
                qa[ks][1] = val1 ? *reinterpret_cast<const unsigned *>(q1 + ks * 16) : 0u;
                qa[ks][2] = val0 ? *reinterpret_cast<const unsigned *>(q0 + ks * 16 + 8) : 0u;
                qa[ks][3] = val1 ? *reinterpret_cast<const unsigned *>(q1 + ks * 16 + 8) : 0u;
            }
        }
        // first sweep: each row's largest score (the scale is positive and rounding is monotonic, so the
        // largest scaled score is the scaled largest score)
        float x0 = -INFINITY, x1 = -INFINITY;
        for (int s = 0; s < ns; ++s) {
            if (!mbar_wait(&full[slot], ph, a.status, DEV_TIMEOUT_LOAD, &s_abort)) return;
            const uint32_t kaddr = smem_u32(ring + (size_t)slot * LY::UNIT) + koff;
            const int k0 = s * ATT_SPLIT;
#pragma unroll 1
            for (int c0 = 0; c0 < ATT_SPLIT && k0 + c0 <= wlast; c0 += 32) {
                float sc[4][4];
                attn_scores<DH>(kaddr + c0 * 128, qa, sc);
                if (k0 + c0 + 31 <= wall) {
#pragma unroll
                    for (int nt = 0; nt < 4; ++nt) {
                        x0 = fmaxf(x0, fmaxf(sc[nt][0], sc[nt][1]));
                        x1 = fmaxf(x1, fmaxf(sc[nt][2], sc[nt][3]));
                    }
                } else {
#pragma unroll
                    for (int nt = 0; nt < 4; ++nt)
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const int kp = k0 + c0 + nt * 8 + 2 * tq + e;
                            x0 = fmaxf(x0, kp <= lim0 ? sc[nt][e] : -INFINITY);
                            x1 = fmaxf(x1, kp <= lim1 ? sc[nt][2 + e] : -INFINITY);
                        }
                }
            }
            __syncwarp();
            if (lane == 0) mbarrier_arrive_one(&empty[slot]);
            if (++slot == RA_UNITS) slot = 0, ph ^= 1;
        }
        x0 = fmaxf(x0, __shfl_xor_sync(0xffffffffu, x0, 1));
        x0 = fmaxf(x0, __shfl_xor_sync(0xffffffffu, x0, 2));
        x1 = fmaxf(x1, __shfl_xor_sync(0xffffffffu, x1, 1));
        x1 = fmaxf(x1, __shfl_xor_sync(0xffffffffu, x1, 2));
        x0 = __fmul_rn(x0, scale);
        x1 = __fmul_rn(x1, scale);
        // second sweep: partial results in key order, added with their weights relative to x0 / x1
        float num[DT][4], den0 = 0.f, den1 = 0.f;
#pragma unroll
        for (int dt = 0; dt < DT; ++dt) num[dt][0] = num[dt][1] = num[dt][2] = num[dt][3] = 0.f;
        for (int s = 0; s < ns; ++s) {
            const int kslot = slot;
            if (!mbar_wait(&full[slot], ph, a.status, DEV_TIMEOUT_LOAD, &s_abort)) return;
            if (++slot == RA_UNITS) slot = 0, ph ^= 1;
            const int vslot = slot;
            if (!mbar_wait(&full[slot], ph, a.status, DEV_TIMEOUT_LOAD, &s_abort)) return;
            if (++slot == RA_UNITS) slot = 0, ph ^= 1;
            const uint32_t kaddr = smem_u32(ring + (size_t)kslot * LY::UNIT) + koff;
            const uint32_t vaddr = smem_u32(ring + (size_t)vslot * LY::UNIT) + voff;
            const int k0 = s * ATT_SPLIT;
#pragma unroll 1
            for (int kb = 0; kb < ATT_SPLIT && k0 + kb <= wlast; kb += HALF) {
                float m0 = -INFINITY, m1 = -INFINITY, l0 = 0.f, l1 = 0.f;
                float oc[DT][4];
#pragma unroll
                for (int dt = 0; dt < DT; ++dt) oc[dt][0] = oc[dt][1] = oc[dt][2] = oc[dt][3] = 0.f;
#pragma unroll 1
                for (int c0 = kb; c0 < kb + HALF && k0 + c0 <= wlast; c0 += 32) {
                    float sc[4][4];
                    attn_scores<DH>(kaddr + c0 * 128, qa, sc);
                    const bool all = k0 + c0 + 31 <= wall;  // (uniform) no key to mask
                    float c0m = -INFINITY, c1m = -INFINITY;
#pragma unroll
                    for (int nt = 0; nt < 4; ++nt)
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            const int kp = k0 + c0 + nt * 8 + 2 * tq + e;
                            sc[nt][e] = all || kp <= lim0 ? __fmul_rn(sc[nt][e], scale) : -INFINITY;
                            sc[nt][2 + e] = all || kp <= lim1 ? __fmul_rn(sc[nt][2 + e], scale) : -INFINITY;
                            c0m = fmaxf(c0m, sc[nt][e]);
                            c1m = fmaxf(c1m, sc[nt][2 + e]);
                        }
                    c0m = fmaxf(c0m, __shfl_xor_sync(0xffffffffu, c0m, 1));
                    c0m = fmaxf(c0m, __shfl_xor_sync(0xffffffffu, c0m, 2));
                    c1m = fmaxf(c1m, __shfl_xor_sync(0xffffffffu, c1m, 1));
                    c1m = fmaxf(c1m, __shfl_xor_sync(0xffffffffu, c1m, 2));
                    const float n0 = fmaxf(m0, c0m), n1 = fmaxf(m1, c1m);
                    if (__any_sync(0xffffffffu, (n0 != m0 && m0 != -INFINITY) || (n1 != m1 && m1 != -INFINITY))) {
                        const float a0 = m0 == -INFINITY ? 0.f : __expf(m0 - n0), a1 = m1 == -INFINITY ? 0.f : __expf(m1 - n1);
                        l0 = __fmul_rn(l0, a0);
                        l1 = __fmul_rn(l1, a1);
#pragma unroll
                        for (int dt = 0; dt < DT; ++dt) {
                            oc[dt][0] = __fmul_rn(oc[dt][0], a0);
                            oc[dt][1] = __fmul_rn(oc[dt][1], a0);
                            oc[dt][2] = __fmul_rn(oc[dt][2], a1);
                            oc[dt][3] = __fmul_rn(oc[dt][3], a1);
                        }
                    }
                    const float z0 = n0 == -INFINITY ? 0.f : n0, z1 = n1 == -INFINITY ? 0.f : n1;
                    m0 = n0;
                    m1 = n1;
#pragma unroll
                    for (int nt = 0; nt < 4; ++nt)
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            sc[nt][e] = __expf(sc[nt][e] - z0);  // (0 for a masked score)
                            sc[nt][2 + e] = __expf(sc[nt][2 + e] - z1);
                            l0 += sc[nt][e];
                            l1 += sc[nt][2 + e];
                        }
#pragma unroll
                    for (int kstep = 0; kstep < 2; ++kstep) {
                        uint32_t pa[4];
                        pa[0] = pack_bf162(sc[2 * kstep][0], sc[2 * kstep][1]);
                        pa[1] = pack_bf162(sc[2 * kstep][2], sc[2 * kstep][3]);
                        pa[2] = pack_bf162(sc[2 * kstep + 1][0], sc[2 * kstep + 1][1]);
                        pa[3] = pack_bf162(sc[2 * kstep + 1][2], sc[2 * kstep + 1][3]);
                        // V of keys at or past T: whatever the page or the ring held, so zero (see attn_split)
                        const int kst = k0 + c0 + kstep * 16;
                        uint32_t ma = 0xFFFFFFFFu, mb = 0xFFFFFFFFu;
                        if (kst + 16 > T) {
                            const int ka = kst + 2 * tq;
                            ma = (ka < T ? 0x0000FFFFu : 0u) | (ka + 1 < T ? 0xFFFF0000u : 0u);
                            mb = (ka + 8 < T ? 0x0000FFFFu : 0u) | (ka + 9 < T ? 0xFFFF0000u : 0u);
                        }
                        // (pages past the CTA's last visible key were not loaded)
                        const int lastpg = (last / PAGE + 1) * PAGE;
                        if (kst >= lastpg) ma = mb = 0u;
                        attn_pv<DH>(vaddr + (c0 + kstep * 16) * 128, pa, ma, mb, oc);
                    }
                }
                l0 += __shfl_xor_sync(0xffffffffu, l0, 1);
                l0 += __shfl_xor_sync(0xffffffffu, l0, 2);
                l1 += __shfl_xor_sync(0xffffffffu, l1, 1);
                l1 += __shfl_xor_sync(0xffffffffu, l1, 2);
                if (l0 > 0.f) {  // (else the row saw no key in this partial result)
                    const float wt = __expf(m0 - x0);
                    den0 = __fadd_rn(den0, __fmul_rn(wt, l0));
#pragma unroll
                    for (int dt = 0; dt < DT; ++dt) {
                        num[dt][0] = __fadd_rn(num[dt][0], __fmul_rn(wt, oc[dt][0]));
                        num[dt][1] = __fadd_rn(num[dt][1], __fmul_rn(wt, oc[dt][1]));
                    }
                }
                if (l1 > 0.f) {
                    const float wt = __expf(m1 - x1);
                    den1 = __fadd_rn(den1, __fmul_rn(wt, l1));
#pragma unroll
                    for (int dt = 0; dt < DT; ++dt) {
                        num[dt][2] = __fadd_rn(num[dt][2], __fmul_rn(wt, oc[dt][2]));
                        num[dt][3] = __fadd_rn(num[dt][3], __fmul_rn(wt, oc[dt][3]));
                    }
                }
            }
            __syncwarp();
            if (lane == 0) {
                mbarrier_arrive_one(&empty[kslot]);
                mbarrier_arrive_one(&empty[vslot]);
            }
        }
        if (val0) {
            bf16 *dst = a.attn + ((size_t)(sg.row0 + i0) * dm.Hq + h0) * DH + 2 * tq;
#pragma unroll
            for (int dt = 0; dt < DT; ++dt)
                *reinterpret_cast<uint32_t *>(dst + dt * 8) = pack_bf162(__fdiv_rn(num[dt][0], den0), __fdiv_rn(num[dt][1], den0));
        }
        if (val1) {
            bf16 *dst = a.attn + ((size_t)(sg.row0 + i1) * dm.Hq + h1) * DH + 2 * tq;
#pragma unroll
            for (int dt = 0; dt < DT; ++dt)
                *reinterpret_cast<uint32_t *>(dst + dt * 8) = pack_bf162(__fdiv_rn(num[dt][2], den1), __fdiv_rn(num[dt][3], den1));
        }
    }
}

// final RMSNorm of read-out row r: the last row of segment ro[r]
__global__ void __launch_bounds__(RW_THREADS) k_rows_final(const __grid_constant__ RowsArgs a, const int *ro, int n_ro,
                                                           const bf16 *__restrict__ gain, bf16 *x_ro) {
    const int lane = threadIdx.x & 31, H = a.dm.H, nt = H / TILE_ROWS;
    const int r = blockIdx.x * (RW_THREADS / 32) + (threadIdx.x >> 5);
    pdl_begin();
    if (r >= n_ro) return;
    const RowSeg sg = a.segs[ro[r]];
    const uint2 *hp = reinterpret_cast<const uint2 *>(a.h + (size_t)(sg.row0 + sg.n - 1) * H) + lane;
    float sum = 0.f;
    for (int t = 0; t < nt; ++t) {
        const uint2 hv = hp[t * 32];
        const __nv_bfloat162 *h2 = reinterpret_cast<const __nv_bfloat162 *>(&hv);
        const float2 p = __bfloat1622float2(h2[0]), q = __bfloat1622float2(h2[1]);
        const float v[4] = {p.x, p.y, q.x, q.y};
        float s = __fmul_rn(v[0], v[0]);
#pragma unroll
        for (int e = 1; e < 4; ++e) s = __fadd_rn(s, __fmul_rn(v[e], v[e]));
        s = warp_sum_butterfly(s);
        sum = t == 0 ? s : __fadd_rn(sum, s);
    }
    const float rs = rms_scale(sum, H, a.dm.eps);
    for (int t = 0; t < nt; ++t)
        reinterpret_cast<uint2 *>(x_ro + (size_t)r * H)[t * 32 + lane] =
            norm4(hp[t * 32], reinterpret_cast<const uint2 *>(gain)[t * 32 + lane], rs);
}

// ------------------------------------------------------------------ host side

cudaError_t configure_rows_kernels() {
    cudaError_t e = cudaFuncSetAttribute(k_rows_attn<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, RaLayout<128>::TOTAL);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_rows_attn<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, RaLayout<64>::TOTAL);
    return e;
}

static int warp_blocks(long warps, int max_ctas) {
    const long b = (warps + RW_THREADS / 32 - 1) / (RW_THREADS / 32);
    return (int)std::min<long>(b, max_ctas > 0 ? max_ctas : 1 << 30);
}

int rows_attn_tile() { return 16 * RA_WARPS; }

cudaError_t launch_rows_embed(const RowsArgs &a, const int *ids, const void *embed_tiled, const void *gain, cudaStream_t st) {
    return launch_pdl(k_rows_embed, warp_blocks(a.M, a.max_ctas), RW_THREADS, 0, st, a, ids,
                      static_cast<const bf16 *>(embed_tiled), static_cast<const bf16 *>(gain));
}

cudaError_t launch_rows_norm(const RowsArgs &a, const void *gain, cudaStream_t st) {
    return launch_pdl(k_rows_norm, warp_blocks(a.M, a.max_ctas), RW_THREADS, 0, st, a, static_cast<const bf16 *>(gain));
}

cudaError_t launch_rows_rope(const RowsArgs &a, int layer, const void *q_norm, const void *k_norm, const float2 *rope_cs,
                             cudaStream_t st) {
    const int grid = a.max_ctas > 0 ? std::min(a.M, a.max_ctas) : a.M;
    const bf16 *qn = static_cast<const bf16 *>(q_norm), *kn = static_cast<const bf16 *>(k_norm);
    return launch_pdl(a.dm.d == 128 ? k_rows_rope<128> : k_rows_rope<64>, grid, RW_THREADS, 0, st, a, layer, qn, kn, rope_cs);
}

cudaError_t launch_rows_attn(const RowsArgs &a, const CUtensorMap &kmap, const CUtensorMap &vmap, int layer,
                             const RowsAttn *work, int n_work, cudaStream_t st) {
    const int grid = a.max_ctas > 0 ? std::min(n_work, a.max_ctas) : n_work;
    return a.dm.d == 128 ? launch_pdl(k_rows_attn<128>, grid, RA_THREADS, RaLayout<128>::TOTAL, st, kmap, vmap, a, layer, work, n_work)
                         : launch_pdl(k_rows_attn<64>, grid, RA_THREADS, RaLayout<64>::TOTAL, st, kmap, vmap, a, layer, work, n_work);
}

cudaError_t launch_rows_final(const RowsArgs &a, const int *ro, int n_ro, const void *gain, void *x_ro, cudaStream_t st) {
    return launch_pdl(k_rows_final, (n_ro + RW_THREADS / 32 - 1) / (RW_THREADS / 32), RW_THREADS, 0, st, a, ro, n_ro,
                      static_cast<const bf16 *>(gain), static_cast<bf16 *>(x_ro));
}

}  // namespace pbd
