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
// 4l..4l+3, as in reduce_qkv (pass_kernel.cu).  Bound by issue slots (66% of them) and the loads' latency, not by
// the 2 x 8 bytes a lane and tile: the row's loads go out before its position is looked up, and one lane
// evaluates the root and divisions of each tile's 1/rms (4096 rows: 28 us without either, 24.5 with
// both; 64 registers for four blocks an SM: at 74 registers 26.7, at 40 spills, 27).
template <int DH>
__global__ void __launch_bounds__(RW_THREADS, 4) k_rows_rope(const __grid_constant__ RowsArgs a, int layer,
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
        uint2 raw[U] = {};
        auto load = [&](int t0) {
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const int ft = (t0 + u * (RW_THREADS / 32)) * TILE_ROWS;
                if (ft < qw + 2 * kvw) raw[u] = *reinterpret_cast<const uint2 *>(a.qkv + (size_t)m * (qw + 2 * kvw) + ft + 4 * lane);
            }
        };
        load(warp);  // (on its way before the row's position is looked up)
        const RowSeg sg = a.segs[row_seg(a, m)];
        const int pos = sg.pos0 + m - sg.row0;
        const float4 *c4 = reinterpret_cast<const float4 *>(rope_cs + (size_t)pos * (DH / 2) + (e0 % (DH / 2)));
        const float4 ca = __ldg(c4), cb = __ldg(c4 + 1);
        const float cs[4] = {ca.x, ca.z, cb.x, cb.z}, sn[4] = {ca.y, ca.w, cb.y, cb.w};
        const size_t slot = ((size_t)layer * a.kv.n_pages + a.kv.page_table[sg.seq * a.kv.pages_per_seq + pos / PAGE]) * dm.Hkv;
        for (int t0 = warp; t0 < nq; t0 += U * (RW_THREADS / 32)) {
            if (t0 != warp) load(t0);
            // the tiles' 1/rms: lane u of a head evaluates tile u's (the root and divisions are as long as the rest)
            float mine = 0.f;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                const float2 ya = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&raw[u].x));
                const float2 yb = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&raw[u].y));
                const float y[4] = {ya.x, ya.y, yb.x, yb.y};
                float ss = __fmul_rn(y[0], y[0]);
#pragma unroll
                for (int j = 1; j < 4; ++j) ss = __fadd_rn(ss, __fmul_rn(y[j], y[j]));
#pragma unroll
                for (int off = LPH / 2; off >= 1; off >>= 1) ss = __fadd_rn(ss, __shfl_xor_sync(0xffffffffu, ss, off));
                if ((lane & (U - 1)) == u) mine = ss;
            }
            const float rs_of = rms_scale(mine, DH, dm.eps);
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
                    const float rs = __shfl_sync(0xffffffffu, rs_of, (lane & ~(LPH - 1)) | u);
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
// One CTA: 128 (row, head) pairs of one sequence's segment and KV head against the cached keys up to the last
// row's position, in the pass kernel's partition: 128-key splits, each one or two partial results of HALF
// keys computed in 32-key chunks with a running maximum, combined in key order relative to the row's
// overall maximum.  The pass kernel stores the partial results and merges them afterwards; here a first
// sweep over the keys finds the overall maximum (scores only), and the second sweep computes each partial
// result and adds it to the row's sums at once, in registers.  One more QK^T per key replaces 520 bytes
// of partial results written and read back per (row, head, partial).
//
// Scores and P V are tcgen05 MMAs: over one K range and in one order of K steps their fp32 sums came out bit for bit
// as mma.sync's (0 of 1.3 M sums differed, over normal, wide-range and probability operands), so the results
// stay the decoding passes'.  Columns of tensor memory: scores of 64-key units [0, 256) in the first
// sweep (four buffers) and [0, 128) in the second (two), P over the scores that it came from (bf16, the A
// operand), the partial result [128, 256).
//
// Roles: warps 0-3 one thread per pair (scores to probabilities, running rescale, sums); warp 4 streams K, then K
// and V, one tiled TMA per 16-token page and 64-dim half; warp 5 issues the MMAs.  One tile keeps the tensor core
// waiting for the softmax and the other way round, so two CTAs share an SM.  The first sweep runs from the
// last unit to the first: the scores of units 0 and 1 are then still there for the second.
//
// Bound: a 32-key chunk is a chain of ~1600 cycles (scores out of tensor memory and to probabilities 620, waits
// 180, rescale or merge 500, P back and handed over 190); two CTAs fill 56% of the issue slots and 28% of
// the tensor core's time.  4096 rows of the 0.6B shape: 165 us a layer; 352 with mma.sync, whose own rate
// would take 176.  725 rows: 34 us against 41.
constexpr int RA_PAIRS = 128;
constexpr int RA_KEYS = 64;      // keys of a unit
constexpr int RA_RING = 4;       // units of K or V in flight
constexpr int RA_THREADS = 256;  // (the second warpgroup has two warps with work)

template <int DH>
struct RaLayout {
    static constexpr int SUB = RA_KEYS * 128;  // 64 keys x 64 dims, 128-byte swizzle
    static constexpr int UNIT = (DH / 64) * SUB;
    static constexpr int QSUB = RA_PAIRS * 128;
    static constexpr int Q = (DH / 64) * QSUB;
    static constexpr int TOTAL = Q + RA_RING * UNIT + 1024;
};

// ring units of an item of nu units of keys
__device__ __forceinline__ int ra_units(int nu) { return 2 * nu + max(nu - 2, 0); }

struct RaState {
    uint64_t full[RA_RING], empty[RA_RING];  // ring
    uint64_t qfull, qfree;                     // q's place filled, given up
    uint64_t sfull1[4], sempty[4], sfull2[2];  // scores: first sweep, second sweep
    uint64_t pfull, pvdone;                    // P of a chunk stored, its P V done
    uint64_t fin;
    uint32_t tmem_slot;
    int abort;
};

template <int DH>
__global__ void __launch_bounds__(RA_THREADS, 2)
    k_rows_attn(const __grid_constant__ CUtensorMap kmap, const __grid_constant__ CUtensorMap vmap,
                const __grid_constant__ RowsArgs a, int layer, const RowsAttn *__restrict__ work, int n_work) {
    using LY = RaLayout<DH>;
    constexpr int KS = DH / 16, SUBS = DH / 64;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *sQ = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t *ring = sQ + LY::Q;
    __shared__ RaState S;
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const Dims &dm = a.dm;
    const int grp = dm.Hq / dm.Hkv;
    if (threadIdx.x == 0) {
        for (int i = 0; i < RA_RING; ++i) {
            mbar_init(&S.full[i], 1);
            mbar_init(&S.empty[i], 1);
        }
        mbar_init(&S.qfull, RA_PAIRS);
        mbar_init(&S.qfree, RA_PAIRS);
        for (int i = 0; i < 4; ++i) {
            mbar_init(&S.sfull1[i], 1);
            mbar_init(&S.sempty[i], RA_PAIRS / 32);
        }
        mbar_init(&S.sfull2[0], 1);
        mbar_init(&S.sfull2[1], 1);
        mbar_init(&S.pfull, RA_PAIRS / 32);
        mbar_init(&S.pvdone, 1);
        mbar_init(&S.fin, 1);
        S.abort = 0;
        fence_mbarrier_init();
        prefetch_tensormap(&kmap);
        prefetch_tensormap(&vmap);
    }
    if (warp == 4) tmem_alloc(&S.tmem_slot, 256);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = S.tmem_slot, tmem_o = tmem + 128;
    // (the work list was uploaded before the pass's first kernel)
    if (warp < 6 && blockIdx.x < n_work) {
        const RowsAttn *wk = work + blockIdx.x;
        asm volatile("prefetch.global.L1 [%0];" ::"l"(wk));
        asm volatile("prefetch.global.L1 [%0];" ::"l"(a.segs + wk->seg));
    }
    pdl_begin();  // (after the allocation: a later kernel's CTA never holds TMEM that this one waits for)
    // an item's last visible key; keys of later pages are not loaded
    auto last_key = [&](const RowsAttn &wk, const RowSeg &sg) { return sg.pos0 + min(sg.n - 1, (wk.q0 + RA_PAIRS - 1) / grp); };
    const int HALF = ATT_SPLIT / a.att_subs;

    // registers: of the launch's 2 x 128 x 128 the second warpgroup keeps 128 x 40, the first takes 128 x 216
    if (warp >= 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
        if (warp == 4) {
            // ---- producer warp: a lane per page and half
            int issued = 0;
            bool ok = true;
            // this pass's own K/V were written by generic stores of an earlier kernel
            fence_proxy_async_global();
            for (int w = blockIdx.x; ok && w < n_work; w += gridDim.x) {
                const RowsAttn wk = work[w];
                const RowSeg sg = a.segs[wk.seg];
                const int last = last_key(wk, sg), nu = last / RA_KEYS + 1;
                for (int i = 0; i < ra_units(nu); ++i) {  // K of every unit, last to first; then V 0, V 1, K 2, V 2, K 3, V 3 ...
                    const int j = i - nu, slot = issued % RA_RING;
                    const bool v = j == 0 || (j > 0 && (j & 1));
                    const int u = j < 0 ? nu - 1 - i : (v ? (j + 1) >> 1 : (j >> 1) + 1);
                    if (!mbar_wait(&S.empty[slot], ((issued / RA_RING) & 1) ^ 1, a.status, DEV_TIMEOUT_SLOT, &S.abort)) ok = false;
                    if (!(ok = __all_sync(0xffffffffu, ok))) break;
                    const int npg = min(RA_KEYS / PAGE, last / PAGE - u * (RA_KEYS / PAGE) + 1);
                    if (lane == 0) mbar_arrive_expect_tx(&S.full[slot], (uint32_t)(npg * SUBS * PAGE * 128));
                    __syncwarp();
                    if (lane < npg * SUBS) {
                        const int p = lane / SUBS, sub = lane % SUBS;
                        const int page = a.kv.page_table[sg.seq * a.kv.pages_per_seq + u * (RA_KEYS / PAGE) + p];
                        tma_load_2d(ring + slot * LY::UNIT + sub * LY::SUB + p * PAGE * 128, v ? &vmap : &kmap, sub * 64,
                                    ((layer * a.kv.n_pages + page) * dm.Hkv + wk.g) * PAGE, &S.full[slot]);
                    }
                    ++issued;
                }
            }
            if (*(volatile int *)&S.abort)  // error path: the copies in flight get a bounded chance to land
                for (int h = issued > RA_RING ? issued - RA_RING : 0; h < issued; ++h)
                    if (!mbar_wait(&S.full[h % RA_RING], (h / RA_RING) & 1, nullptr, 0, nullptr)) break;  // (all had this second)
        } else if (warp == 5 && elect_one()) {
            // ---- MMA warp
            const uint32_t ids = idesc_bf16_f32(128, RA_KEYS), ido = idesc_bf16_f32(128, DH) | IDESC_B_MN;
            const uint64_t qd = sw128_kmajor_desc(sQ);
            int used = 0;  // ring units
            uint32_t ph = 0;  // phase bits: 0-3 sempty, 4 pfull, 5 qfull
            bool ok = true;
            auto wait = [&](uint64_t *bar, int bit) {
                ok = ok && mbar_wait(bar, (ph >> bit) & 1u, a.status, DEV_TIMEOUT_MMA, &S.abort);
                ph ^= 1u << bit;
                return ok;
            };
            auto unit = [&]() {  // the next ring unit, once it has landed
                const int slot = used % RA_RING;
                ok = ok && mbar_wait(&S.full[slot], (used / RA_RING) & 1, a.status, DEV_TIMEOUT_LOAD, &S.abort);
                ++used;
                return slot;
            };
            auto scores = [&](uint32_t col, uint64_t *bar) {
                const int slot = unit();
                if (!ok) return;
                tc_fence_after();
                const uint64_t kd = sw128_kmajor_desc(ring + slot * LY::UNIT);
#pragma unroll
                for (int ks = 0; ks < KS; ++ks)
                    mma_bf16_ss(tmem + col, qd + (uint64_t)((ks >> 2) * LY::QSUB / 16 + 2 * (ks & 3)),
                                kd + (uint64_t)((ks >> 2) * LY::SUB / 16 + 2 * (ks & 3)), ids, ks != 0);
                mma_commit(&S.empty[slot]);
                mma_commit(bar);
            };
            for (int w = blockIdx.x; ok && w < n_work; w += gridDim.x) {
                const RowsAttn wk = work[w];
                const RowSeg sg = a.segs[wk.seg];
                const int last = last_key(wk, sg), nu = last / RA_KEYS + 1;
                if (!wait(&S.qfull, 5)) break;
                for (int u = nu - 1; ok && u >= 0; --u) {
                    if (u + 4 < nu) wait(&S.sempty[u & 3], u & 3);
                    scores((u & 3) * RA_KEYS, &S.sfull1[u & 3]);
                }
                for (int u = 0; ok && u < min(nu, 4); ++u) wait(&S.sempty[u & 3], u & 3);
                for (int u = 0; ok && u < nu; ++u) {
                    int vslot = 0;
                    for (int cc = 0; cc < 2; ++cc) {
                        const int k = u * RA_KEYS + cc * 32;
                        if (k > last) break;
                        // (every thread of the softmax saw the P V before this one done: the other scores'
                        // columns are free)
                        if (!wait(&S.pfull, 4)) break;
                        if (cc == 0) vslot = unit();
                        if (!ok) break;
                        tc_fence_after();
                        const uint64_t vd = sw128_mnmajor_desc(ring + vslot * LY::UNIT, LY::SUB);
#pragma unroll
                        for (int j = 0; j < 2; ++j)
                            if (k + j * PAGE <= last)
                                mma_bf16_ts(tmem_o, tmem + (u & 1) * RA_KEYS + cc * 32 + j * 8,
                                            vd + (uint64_t)((cc * 2 + j) * PAGE * 128 >> 4), ido, j != 0 || (k & (HALF - 1)) != 0);
                        mma_commit(&S.pvdone);
                        if (cc == 0 && u >= 1 && u + 1 < nu) scores(((u + 1) & 1) * RA_KEYS, &S.sfull2[(u + 1) & 1]);
                    }
                    if (ok) mma_commit(&S.empty[vslot]);
                }
            }
            mma_commit(&S.fin);  // also on the error path: every MMA issued completes before TMEM goes
            mbar_wait(&S.fin, 0, nullptr, 0, nullptr);
        }
    } else {
        // ---- softmax: thread t the pair q0 + t (tensor memory lane t)
        asm volatile("setmaxnreg.inc.sync.aligned.u32 216;");
        const uint32_t tl = tmem + ((uint32_t)(warp * 32) << 16), to = tl + 128;
        const float scale = a.att_scale;
        uint32_t ph = 0;  // phase bits: 0-3 sfull1, 4-5 sfull2, 6 pvdone, 7 qfree
        int units = 0;    // ring units before this item's
        auto wait = [&](uint64_t *bar, int bit) {
            bool ok = false;
            for (int t = 0; t < 4096 && !ok; ++t) ok = mbar_test_wait(smem_u32(bar), (ph >> bit) & 1u);
            if (!ok) ok = mbar_wait(bar, (ph >> bit) & 1u, a.status, DEV_TIMEOUT_MMA, &S.abort);
            ph ^= 1u << bit;
            return __all_sync(0xffffffffu, ok) != 0;
        };
        bool ok = true;
        for (int w = blockIdx.x; ok && w < n_work; w += gridDim.x) {
            const RowsAttn wk = work[w];
            const RowSeg sg = a.segs[wk.seg];
            const int last = last_key(wk, sg), nu = last / RA_KEYS + 1, T = sg.pos0 + sg.n, QV = sg.n * grp;
            if (w != blockIdx.x && !(ok = wait(&S.qfree, 7))) break;  // (the last item's sums were staged there)
            for (int q = threadIdx.x; q < RA_PAIRS * (DH / 8); q += RA_PAIRS) {
                const int r = q / (DH / 8), c = q % (DH / 8), qv = wk.q0 + r;
                if (qv < QV)
                    cp_async16(sQ + (c >> 3) * LY::QSUB + r * 128 + (((c & 7) ^ (r & 7)) << 4),
                               a.q + ((size_t)(sg.row0 + qv / grp) * dm.Hq + wk.g * grp + qv % grp) * DH + c * 8);
            }
            cp_async_commit();
            cp_async_wait_all();
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            mbarrier_arrive_one(&S.qfull);
            const int qv = wk.q0 + threadIdx.x;
            const bool val = qv < QV;
            const int i = val ? qv / grp : 0, h = wk.g * grp + (val ? qv % grp : 0);
            const int lim = val ? sg.pos0 + i : -1;  // last visible key
            // the warp's last visible key (-1: no pairs), and the last key that all its pairs see
            const int wq0 = wk.q0 + warp * 32;
            const int wlast = wq0 < QV ? sg.pos0 + min(sg.n - 1, (wq0 + 31) / grp) : -1;
            const int wall = wq0 + 31 < QV ? sg.pos0 + wq0 / grp : -1;
            // first sweep: the largest score (the scale is positive and rounding is monotonic, so the
            // largest scaled score is the scaled largest score)
            float x = -INFINITY;
            for (int u = nu - 1; u >= 0; --u) {
                if (!(ok = wait(&S.sfull1[u & 3], u & 3))) break;
                tc_fence_after();
                const int k0 = u * RA_KEYS;
#pragma unroll 1
                for (int k = k0; k < k0 + RA_KEYS && k <= wlast; k += 32) {
                    uint32_t v[32];
                    tmem_ld_32cols(tl + (u & 3) * RA_KEYS + (k - k0), v);
                    tmem_ld_wait();
                    float y[4] = {x, x, x, x};
                    if (k + 31 <= wall) {
#pragma unroll
                        for (int e = 0; e < 32; ++e) y[e & 3] = fmaxf(y[e & 3], __uint_as_float(v[e]));
                    } else {
#pragma unroll
                        for (int e = 0; e < 32; ++e) y[e & 3] = fmaxf(y[e & 3], k + e <= lim ? __uint_as_float(v[e]) : -INFINITY);
                    }
                    x = fmaxf(fmaxf(y[0], y[1]), fmaxf(y[2], y[3]));
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbarrier_arrive_one(&S.sempty[u & 3]);
                __syncwarp();
            }
            if (!ok) break;
            x = __fmul_rn(x, scale);
            // second sweep: partial results in key order, added with their weights relative to x
            F2 num[DH / 2];
            float den = 0.f;
#pragma unroll
            for (int d = 0; d < DH / 2; ++d) num[d] = f2(0.f, 0.f);
            // running maximum and sum of the partial result; l[j]: the keys 2j, 2j + 1 (mod 8)
            float m = -INFINITY, l[4] = {0.f, 0.f, 0.f, 0.f};
            // (the last iteration only merges)
#pragma unroll 1
            for (int k = 0;; k += 32) {
                const int u = k / RA_KEYS;
                const uint32_t cols = tl + (u & 1) * RA_KEYS + (k & 32);
                const bool more = k <= last, first = !more || (k & (HALF - 1)) == 0;
                const float pm = m, pl = __fadd_rn(__fadd_rn(l[0], l[1]), __fadd_rn(l[2], l[3]));
                bool grow = false;
                float sc = 0.f;
                uint32_t p[16];
                if (more) {
                    if (u >= 2 && (k & 32) == 0 && !(ok = wait(&S.sfull2[u & 1], 4 + (u & 1)))) break;
                    tc_fence_after();
                    uint32_t v[32];
                    tmem_ld_32cols(cols, v);
                    if (first) {
                        m = -INFINITY;
                        l[0] = l[1] = l[2] = l[3] = 0.f;
                    }
                    tmem_ld_wait();
                    if (k + 31 > wall)
#pragma unroll
                        for (int e = 0; e < 32; ++e)
                            if (k + e > lim) v[e] = 0xff800000u;  // -infinity (the scale is positive)
                    float cm[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
                    for (int e = 0; e < 32; e += 2) {
                        const float y0 = __fmul_rn(__uint_as_float(v[e]), scale), y1 = __fmul_rn(__uint_as_float(v[e + 1]), scale);
                        v[e] = __float_as_uint(y0);
                        v[e + 1] = __float_as_uint(y1);
                        cm[(e >> 1) & 3] = fmaxf(fmaxf(cm[(e >> 1) & 3], y0), y1);
                    }
                    const float n = fmaxf(m, fmaxf(fmaxf(cm[0], cm[1]), fmaxf(cm[2], cm[3])));
                    grow = __any_sync(0xffffffffu, n != m && m != -INFINITY);
                    sc = m == -INFINITY ? 0.f : __expf(m - n);
                    if (grow)
#pragma unroll
                        for (int j = 0; j < 4; ++j) l[j] = __fmul_rn(l[j], sc);
                    const float z = n == -INFINITY ? 0.f : n;
                    m = n;
#pragma unroll
                    for (int e = 0; e < 32; e += 2) {
                        const float p0 = __expf(__uint_as_float(v[e]) - z), p1 = __expf(__uint_as_float(v[e + 1]) - z);  // (0 if masked)
                        l[(e >> 1) & 3] += p0;
                        l[(e >> 1) & 3] += p1;
                        p[e >> 1] = pack_bf162(p0, p1);
                    }
                }
                if (k > 0) {
                    if (!(ok = wait(&S.pvdone, 6))) break;
                    tc_fence_after();
                    if (first) {
                        // the finished partial result joins the row's sums
                        const float wt = __expf(pm - x);
                        if (pl > 0.f) den = __fadd_rn(den, __fmul_rn(wt, pl));
#pragma unroll
                        for (int d0 = 0; d0 < DH; d0 += 32) {
                            uint32_t o[32];
                            tmem_ld_32cols(to + d0, o);
                            tmem_ld_wait();
                            if (pl > 0.f)  // (else the pair saw no key in this partial result)
#pragma unroll
                                for (int d = 0; d < 16; ++d)
                                    num[d0 / 2 + d] = add2(num[d0 / 2 + d], mul2(wt, __uint_as_float(o[2 * d]), __uint_as_float(o[2 * d + 1])));
                            __syncwarp();
                        }
                    } else if (grow) {
#pragma unroll 1
                        for (int d0 = 0; d0 < DH; d0 += 32) {
                            uint32_t o[32];
                            tmem_ld_32cols(to + d0, o);
                            tmem_ld_wait();
#pragma unroll
                            for (int d = 0; d < 32; d += 2) {
                                const float2 y = unpack2(mulp2(f2(__uint_as_float(o[d]), __uint_as_float(o[d + 1])), f2(sc, sc)));
                                o[d] = __float_as_uint(y.x);
                                o[d + 1] = __float_as_uint(y.y);
                            }
                            tmem_st_32cols(to + d0, o);
                        }
                    }
                }
                if (!more) break;
                tmem_st_16cols(cols, p);
                tmem_st_wait();
                // V of keys at or past T in the last page: whatever the page held, so zero (0 x NaN)
                if (warp == 0 && k + 32 > last && T % PAGE && T < (last / PAGE + 1) * PAGE) {
                    const int vu = units + nu + max(2 * u - 1, 0);
                    uint8_t *vs = ring + (vu % RA_RING) * LY::UNIT;
                    ok = mbar_wait(&S.full[vu % RA_RING], (vu / RA_RING) & 1, a.status, DEV_TIMEOUT_LOAD, &S.abort);
                    if (!(ok = __all_sync(0xffffffffu, ok))) break;
                    const int r0 = T - u * RA_KEYS, nr = (last / PAGE + 1) * PAGE - T;
                    for (int e = lane; e < nr * SUBS * 8; e += 32)
                        *reinterpret_cast<uint4 *>(vs + (e / (nr * 8)) * LY::SUB + (r0 + (e / 8) % nr) * 128 + (e % 8) * 16) =
                            make_uint4(0, 0, 0, 0);
                    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbarrier_arrive_one(&S.pfull);
                __syncwarp();
            }
            if (!ok) break;
            tc_fence_before();
            units += ra_units(nu);
            // Quotients, in a loop out of shared memory (q's place: every MMA has read it) to keep the code short: a short
            // prompt's time is that of fetching it.  The result is the bf16 of the fp32 quotient x / den.
            // The products of x with two numbers around 1 / den bracket that quotient (rounding is
            // monotonic), so where both give one bf16 value it is the result; else (1 in 10^4) it is
            // divided.  __fdiv_rn for all took 5 us a tile: its rare-case branches keep divisions from overlapping.
            constexpr int NC = LY::Q / (RA_PAIRS * 16);  // float4 per pair that fit
            float4 *stage = reinterpret_cast<float4 *>(sQ) + threadIdx.x;
            bf16 *dst = a.attn + ((size_t)(sg.row0 + i) * dm.Hq + h) * DH;
            const bool plain = den > 1e-30f && den < 1e30f;
            const float rc = __frcp_rn(den), rlo = __fmul_rn(rc, 1.f - 0x1p-22f), rhi = __fmul_rn(rc, 1.f + 0x1p-22f);
#pragma unroll
            for (int d0 = 0; d0 < DH; d0 += 4 * NC) {
#pragma unroll
                for (int c = 0; c < NC; ++c) {
                    const float2 y0 = unpack2(num[d0 / 2 + 2 * c]), y1 = unpack2(num[d0 / 2 + 2 * c + 1]);
                    stage[c * RA_PAIRS] = make_float4(y0.x, y0.y, y1.x, y1.y);
                }
                if (val)
#pragma unroll 1
                    for (int c = 0; c < NC; c += 2) {
                        const float4 y0 = stage[c * RA_PAIRS], y1 = stage[(c + 1) * RA_PAIRS];
                        const float y[8] = {y0.x, y0.y, y0.z, y0.w, y1.x, y1.y, y1.z, y1.w};
                        uint32_t o[4];
                        bool same = plain;
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            o[e] = pack_bf162(__fmul_rn(y[2 * e], rlo), __fmul_rn(y[2 * e + 1], rlo));
                            same = same && o[e] == pack_bf162(__fmul_rn(y[2 * e], rhi), __fmul_rn(y[2 * e + 1], rhi));
                        }
                        if (!same)
#pragma unroll
                            for (int e = 0; e < 4; ++e) o[e] = pack_bf162(__fdiv_rn(y[2 * e], den), __fdiv_rn(y[2 * e + 1], den));
                        *reinterpret_cast<uint4 *>(dst + d0 + 4 * c) = make_uint4(o[0], o[1], o[2], o[3]);
                    }
            }
            mbarrier_arrive_one(&S.qfree);
        }
        tc_fence_before();
    }
    __syncwarp();
    __syncthreads();
    if (warp == 4) tmem_dealloc(tmem, 256);
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

template <int DH>
static cudaError_t configure_rows_attn() {
    const void *f = (const void *)k_rows_attn<DH>;
    const cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, RaLayout<DH>::TOTAL);
    return e != cudaSuccess ? e : cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
}

cudaError_t configure_rows_kernels() {
    const cudaError_t e = configure_rows_attn<128>();
    return e != cudaSuccess ? e : configure_rows_attn<64>();
}

static int warp_blocks(long warps, int max_ctas) {
    const long b = (warps + RW_THREADS / 32 - 1) / (RW_THREADS / 32);
    return (int)std::min<long>(b, max_ctas > 0 ? max_ctas : 1 << 30);
}

int rows_attn_tile() { return RA_PAIRS; }

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
