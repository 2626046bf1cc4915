// steps.cu -- a decoding pass (draft, verify, plain decoding) as a chain of small dependent kernels.
//
// A layer is five kernels: q|k|v (+ QK-norm, RoPE, K/V write), attention, o (+ residual), gate|up (+ SiLU),
// down (+ residual).  Each is one step of the chain, bound by latency and not by its few megabytes of
// weights, so the design removes what the chain waits for:
//   - A linear's K slices (256 wide, gate|up 512) are one thread-block cluster per 128-feature tile.  A
//     row's fp32 partial sums go through distributed shared memory to the CTA that finishes the row (many
//     rows: it fetches them).  The attention's key splits of a (sequence, KV head) are a cluster too, as
//     long as there are few of them, and merge the same way.
//   - The kernels launch dependent: a CTA sets itself up and requests its weights (or the cached K/V
//     pages) while the step before it still runs, and waits only for its activations.
//
// The arithmetic is the persistent pass kernel's (pass_kernel.cu), operation for operation: K slices and
// their order, key partition, every sum and rounding.  That kernel remains for contexts limited to fewer
// CTAs than SMs and for shapes whose slices or partial results do not fit a cluster; rows.cu computes the
// same for prompts.
//
// 0.6B shape, all layers of one pass (the persistent kernel in brackets), us: verify 758 (1136), draft 959
// (1287), one-row decoding 619 (945) at 512 tokens of context; 880 (1430), 1090 (1579), 731 (1196) at 4096;
// 1609 (3637), 2060 (4080), 846 (1778) for eight sequences of 420 to 1757 tokens.
#include <algorithm>
#include <cmath>

#include "attn.cuh"
#include "common.cuh"
#include "pbd_internal.h"

namespace pbd {

constexpr int ST_HALF = 4;         // 64-wide K atoms per half (256 of K)
constexpr int ST_RANK = 16;        // adapter rank (8 or 16)
constexpr int ST_A_BYTES = 2 * ST_RANK * 128;  // adapter rows of one K atom (gate and up: two ranks)

template <int N>
__device__ __forceinline__ void bar_stagers() {
    asm volatile("bar.sync 1, %0;" ::"n"(N) : "memory");
}

__device__ __forceinline__ float4 add4(float4 a, float4 b) {
    return make_float4(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y), __fadd_rn(a.z, b.z), __fadd_rn(a.w, b.w));
}

// ------------------------------------------------------------------ linear step

struct StepLinState {
    uint64_t wfull[2], xfull[2], hdone, done;
    uint32_t tmem_slot;
    int abort;
    float rs[256];  // 1/rms of each row (normalised operands)
    // the adapter's B rows of the tile, transposed and widened: [rank][128] (a reducing lane reads four features
    // of one rank column at a time)
    float4 bt[ST_RANK * TILE_ROWS / 4];
};

// Sum over the slices, in slice order, of four features of a row or of one adapter row.  PUSH: the slices lie
// `stride` bytes apart in this CTA; otherwise slice s at the same address of CTA s.
__device__ __forceinline__ float4 slice4(uint32_t a, int s, uint32_t stride, bool push) {
    return push ? ld_shared_v4(a + (uint32_t)s * stride) : ld_cluster_v4(map_cta(a, s));
}
__device__ __forceinline__ float4 sum_slices4(uint32_t a, int ks, uint32_t stride, bool push) {
    float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int s0 = 0; s0 < ks; s0 += 4) {
        float4 v[4];
#pragma unroll
        for (int s = 0; s < 4; ++s) v[s] = slice4(a, min(s0 + s, ks - 1), stride, push);
#pragma unroll
        for (int s = 0; s < 4; ++s)
            if (s0 + s < ks) y = s0 + s == 0 ? v[s] : add4(y, v[s]);
    }
    return y;
}
__device__ __forceinline__ float sum_slices(uint32_t a, int ks, uint32_t stride, bool push) {
    float y = 0.f;
    for (int s0 = 0; s0 < ks; s0 += 4) {
        float v[4];
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            const int t = min(s0 + s, ks - 1);
            v[s] = push ? ld_shared(a + (uint32_t)t * stride) : ld_cluster(map_cta(a, t));
        }
#pragma unroll
        for (int s = 0; s < 4; ++s)
            if (s0 + s < ks) y = s0 + s == 0 ? v[s] : __fadd_rn(y, v[s]);
    }
    return y;
}

// y_f += scale * (u . B_f) for two pairs of features f, the products added in rank order.
// lane_ua / lane_ub: lane i holds u_i for the first / second pair of features (at fa, fb in the tile)
__device__ __forceinline__ void add_delta(float (&y)[4], float lane_ua, float lane_ub, int base_b, const float *bt, int fa, int fb,
                                          int r, float scale) {
    F2 a = f2(0.f, 0.f), b = a;
#pragma unroll
    for (int i = 0; i < ST_RANK; ++i) {
        if (i >= r) break;
        const float ua = __shfl_sync(0xffffffffu, lane_ua, i), ub = __shfl_sync(0xffffffffu, lane_ub, base_b + i);
        const float2 ba = *reinterpret_cast<const float2 *>(bt + i * TILE_ROWS + fa);
        const float2 bb = *reinterpret_cast<const float2 *>(bt + i * TILE_ROWS + fb);
        a = add2(a, mul2(ua, ba.x, ba.y));
        b = add2(b, mul2(ub, bb.x, bb.y));
    }
    const float2 da = unpack2(a), db = unpack2(b);
    const float2 ya = unpack2(add2(f2(y[0], y[1]), mul2(scale, da.x, da.y))), yb = unpack2(add2(f2(y[2], y[3]), mul2(scale, db.x, db.y)));
    y[0] = ya.x, y[1] = ya.y, y[2] = yb.x, y[3] = yb.y;
}

// LIN: 0 q|k|v, 1 o, 2 gate|up, 3 down.  Grid (tiles, slices), cluster (1, slices).
// NT threads: warp 0 streams, warp 1 issues the MMAs, warps 2.. stage a normalised operand, warps 4-7 read the
// accumulator, all finish rows.  Dynamic shared memory: W atoms | adapter atoms (AD) | x atoms | partial sums
// (or those in the operands' place).
template <int LIN, bool AD, int DH, int NT>
__global__ void __maxnreg__(NT == 256 ? 104 : 128)
    k_step_linear(const __grid_constant__ StepArgs a, const __grid_constant__ StepLin w) {
    constexpr bool NORM = LIN == 0 || LIN == 2;  // the operand is RMSNorm(h)
    constexpr int STAGERS = NT - 64;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ StepLinState S;
    const Dims &dm = a.dm;
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int tile = blockIdx.x, slice = blockIdx.y, M = a.pd.M, r = dm.r;
    const int ra = w.ring_atoms, x_atom = a.bn * 128;
    uint8_t *sW = base, *sA = base + ra * TILE_BYTES, *sX = sA + (AD ? ra * ST_A_BYTES : 0);
    const int halves = w.katoms / ST_HALF;
    // features of this tile, and the adapter rows that its delta uses: its projection's rank rows (both gate's
    // and up's for gate|up)
    const int qw = dm.Hq * DH, kvw = dm.Hkv * DH, ft = tile * TILE_ROWS;
    const int kind = LIN == 0 ? (ft < qw ? 0 : (ft < qw + kvw ? 1 : 2)) : 0;
    const int ru = LIN == 2 ? 2 * r : r;
    if (threadIdx.x == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(&S.wfull[i], 1);
            mbar_init(&S.xfull[i], 1);
        }
        mbar_init(&S.hdone, 1);
        mbar_init(&S.done, 1);
        S.abort = 0;
        fence_mbarrier_init();
        if (!NORM) prefetch_tensormap(&w.xmap);
    }
    if (warp == 0) tmem_alloc(&S.tmem_slot, w.tmem_cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = S.tmem_slot;
    cluster_arrive();  // (this CTA's shared memory exists: its peers wait for that before they write there)
    pdl_launch();  // (after the allocation: a later kernel's CTA never holds TMEM that this one waits for)

    if (warp == 0 && elect_one()) {
        // ---- weights at once, the second half when it has room; the activations once they are there
        const uint64_t pol = l2_policy_evict_first();
        auto weights = [&](int hf) {
            const int at = (hf * ST_HALF) % ra;
            mbar_arrive_expect_tx(&S.wfull[hf], (uint32_t)(ST_HALF * (TILE_BYTES + (AD ? ru * 128 : 0))));
            const size_t k0 = (size_t)slice * w.katoms + hf * ST_HALF;
            bulk_g2s(sW + at * TILE_BYTES, w.tiles + ((size_t)tile * w.k_tiles + k0) * TILE_BYTES, ST_HALF * TILE_BYTES,
                     &S.wfull[hf], pol);
            if (AD)
                for (int j = 0; j < ST_HALF; ++j)
                    bulk_g2s(sA + (at + j) * ST_A_BYTES,
                             w.tiles + ((size_t)(w.n_main / TILE_ROWS) * w.k_tiles + k0 + j) * TILE_BYTES + kind * r * 128,
                             (uint32_t)(ru * 128), &S.wfull[hf], pol);
        };
        weights(0);
        if (halves == 2 && ra > ST_HALF) weights(1);
        if (!NORM) {
            pdl_wait();
            fence_proxy_async_global();
            mbar_arrive_expect_tx(&S.xfull[0], (uint32_t)(ST_HALF * x_atom));
            for (int j = 0; j < ST_HALF; ++j)
                tma_load_2d(sX + j * x_atom, &w.xmap, (slice * ST_HALF + j) * KT, 0, &S.xfull[0]);
        }
        bool second = halves == 2 && ra > ST_HALF;
        if (halves == 2 && !second && mbar_wait(&S.hdone, 0, a.status, DEV_TIMEOUT_MMA, &S.abort)) {
            weights(1);
            second = true;
        }
        if (*(volatile int *)&S.abort) {  // error path: the copies in flight get a bounded chance to land
            mbar_wait(&S.wfull[0], 0, nullptr, 0, nullptr);
            if (second) mbar_wait(&S.wfull[1], 0, nullptr, 0, nullptr);
            if (!NORM) mbar_wait(&S.xfull[0], 0, nullptr, 0, nullptr);
        }
    } else if (warp == 1 && elect_one()) {
        // ---- MMAs: 16 (and 16 of the adapter) per half
        const uint32_t idesc = idesc_bf16_f32(128, a.bn);
        for (int hf = 0; hf < halves; ++hf) {
            if (!mbar_wait(&S.wfull[hf], 0, a.status, DEV_TIMEOUT_LOAD, &S.abort) ||
                !mbar_wait(&S.xfull[hf], 0, a.status, DEV_TIMEOUT_LOAD, &S.abort))
                break;
            tc_fence_after();
            const int at = (hf * ST_HALF) % ra;
#pragma unroll
            for (int j = 0; j < ST_HALF; ++j) {
                const uint64_t wd = sw128_kmajor_desc(sW + (at + j) * TILE_BYTES), xd = sw128_kmajor_desc(sX + (at + j) * x_atom);
#pragma unroll
                for (int kk = 0; kk < KT / 16; ++kk)
                    mma_bf16_ss(tmem, wd + 2ull * kk, xd + 2ull * kk, idesc, (hf | j | kk) != 0 ? 1u : 0u);
            }
            if (AD)
#pragma unroll
                for (int j = 0; j < ST_HALF; ++j) {
                    // (reads 128 rows from the adapter rows on: what follows them reaches only accumulator
                    // rows that nobody reads)
                    const uint64_t ad = sw128_kmajor_desc(sA + (at + j) * ST_A_BYTES), xd = sw128_kmajor_desc(sX + (at + j) * x_atom);
#pragma unroll
                    for (int kk = 0; kk < KT / 16; ++kk)
                        mma_bf16_ss(tmem + a.bn, ad + 2ull * kk, xd + 2ull * kk, idesc, (hf | j | kk) != 0 ? 1u : 0u);
                }
            if (halves == 2 && hf == 0) mma_commit(&S.hdone);
        }
        mma_commit(&S.done);  // also on the error path: every MMA issued completes before TMEM goes
    } else if (warp >= 2) {
        const int ct = threadIdx.x - 64, c = ct & 31;  // c: the thread's 16-byte chunk column
        uint4 gv[2] = {make_uint4(0, 0, 0, 0), make_uint4(0, 0, 0, 0)};
        if (NORM)
            for (int hf = 0; hf < halves; ++hf)
                gv[hf] = __ldg(reinterpret_cast<const uint4 *>(w.gain + (size_t)(slice * w.katoms + hf * ST_HALF) * KT) + c);
        if (AD) {
            const int cpr = r / 8;
            float *bt = reinterpret_cast<float *>(S.bt);
            for (int q = ct; q < TILE_ROWS * cpr; q += STAGERS) {
                const int j = q % TILE_ROWS, e = q / TILE_ROWS;
                const int f = LIN == 2 ? (j < 64 ? tile * 64 + j : dm.I + tile * 64 + (j - 64)) : ft + j;
                const uint4 v = __ldg(reinterpret_cast<const uint4 *>(w.lora_b + (size_t)f * r) + e);
                const bf16 *x = reinterpret_cast<const bf16 *>(&v);
#pragma unroll
                for (int i = 0; i < 8; ++i) bt[(e * 8 + i) * TILE_ROWS + j] = bf2f(x[i]);
            }
        }
        pdl_wait();
        if (NORM) {
            // ---- operand staging: the rows' chunks straight into the swizzled layout, then normalised in place
            // (as build_b in pass_kernel.cu)
            uint8_t *col = sX + (size_t)(c >> 3) * x_atom;
            auto chunk = [&](int at, int m) { return col + at * x_atom + m * 128 + (((c & 7) ^ (m & 7)) << 4); };
            const bool both = halves == 2 && ra > ST_HALF;  // room for both halves at once
            auto copy = [&](int hf) {
                const bf16 *src = a.h + (size_t)(slice * w.katoms + hf * ST_HALF) * KT + c * 8;
#pragma unroll 1
                for (int m = ct >> 5; m < M; m += STAGERS / 32) cp_async16(chunk((hf * ST_HALF) % ra, m), src + (size_t)m * dm.H);
                cp_async_commit();
            };
            copy(0);
            if (both) copy(1);
            bool ok = true;
            for (int hf = 0; hf < halves; ++hf) {
                const int at = (hf * ST_HALF) % ra;
                if (hf == 1 && !both) {
                    if (!mbar_wait(&S.hdone, 0, a.status, DEV_TIMEOUT_MMA, &S.abort)) ok = false;
                    if (!ok) break;
                    copy(1);
                }
                if (hf == 0) {
                    const int nt = dm.H / TILE_ROWS;
                    for (int m = ct; m < M; m += STAGERS) {
                        const float2 *s = reinterpret_cast<const float2 *>(a.ss + (size_t)m * nt);
                        float sum = 0.f;
                        for (int t0 = 0; t0 < nt; t0 += 8) {
                            float2 v[4];
#pragma unroll
                            for (int u = 0; u < 4; ++u) v[u] = t0 + 2 * u < nt ? __ldcg(s + t0 / 2 + u) : make_float2(0.f, 0.f);
#pragma unroll
                            for (int u = 0; u < 4; ++u) {
                                if (t0 + 2 * u >= nt) break;
                                sum = (t0 + u == 0) ? v[u].x : __fadd_rn(sum, v[u].x);
                                sum = __fadd_rn(sum, v[u].y);
                            }
                        }
                        S.rs[m] = rms_scale(sum, dm.H, dm.eps);
                    }
                }
                if (hf == 0 && both)
                    cp_async_wait_1();
                else
                    cp_async_wait_all();
                if (hf == 0) bar_stagers<STAGERS>();
                const __nv_bfloat162 *g2 = reinterpret_cast<const __nv_bfloat162 *>(&gv[hf]);
#pragma unroll 1
                for (int m = ct >> 5; m < M; m += STAGERS / 32) {
                    uint4 *p = reinterpret_cast<uint4 *>(chunk(at, m));
                    uint4 val = *p;
                    __nv_bfloat162 *v2 = reinterpret_cast<__nv_bfloat162 *>(&val);
                    const float rs = S.rs[m];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float2 f = __bfloat1622float2(v2[e]);
                        v2[e] = __hmul2(g2[e], __floats2bfloat162_rn(__fmul_rn(f.x, rs), __fmul_rn(f.y, rs)));
                    }
                    *p = val;
                }
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                bar_stagers<STAGERS>();
                if (ct == 0) mbarrier_arrive_one(&S.xfull[hf]);
            }
        }
    }
    __syncwarp();

    // what the warp's first row needs besides its sums, on its way early
    const int m_first = slice + warp * w.ks;
    int pos1 = 0, page1 = 0;
    float4 rope1[2] = {make_float4(0.f, 0.f, 0.f, 0.f), make_float4(0.f, 0.f, 0.f, 0.f)};
    uint2 h1 = make_uint2(0, 0);
    auto row_pos = [&](int m) { return a.L[a.pd.b0 + m / a.pd.R] + m % a.pd.R; };
    auto row_page = [&](int m, int pos) {
        return pos / PAGE < a.kv.pages_per_seq ? a.kv.page_table[(a.pd.b0 + m / a.pd.R) * a.kv.pages_per_seq + pos / PAGE] : -1;
    };
    auto row_rope = [&](int pos, float4 (&c)[2]) {
        const float4 *p = reinterpret_cast<const float4 *>(a.rope_cs + (size_t)(pos < a.rope_rows ? pos : 0) * (DH / 2) +
                                                           (4 * (lane % (DH / 4))) % (DH / 2));
        c[0] = __ldg(p);
        c[1] = __ldg(p + 1);
    };
    if (warp < 2) pdl_wait();  // (the warps that have not yet)
    if (m_first < M) {
        if (LIN == 0) {
            pos1 = row_pos(m_first);
            if (kind > 0) page1 = row_page(m_first, pos1);
            if (kind < 2) row_rope(pos1, rope1);
        } else if (LIN != 2) {
            h1 = __ldcg(reinterpret_cast<const uint2 *>(a.h + (size_t)m_first * dm.H + ft) + lane);
        }
    }

    // ---- partial sums: warps 4-7 (and 8-11), a TMEM lane quarter (32 features) each.  PUSH: row m straight to CTA
    // m % slices, which finishes it, as [slice][row / slices][features] behind its ring.  Otherwise (many
    // rows) into the ring's place, every MMA having read its operands, for the peers to read.
    const bool push = w.push != 0;
    const int rpo = (M + w.ks - 1) / w.ks;  // rows per CTA
    float *part = reinterpret_cast<float *>(push ? sX + ra * x_atom : base);
    float *part_u = part + (push ? w.ks * rpo : M) * TILE_ROWS;
    const uint32_t pa = smem_u32(part), pu = smem_u32(part_u);
    cluster_wait();
    constexpr int MOVERS = NT / 128 > 2 ? 2 : 1;  // warps per lane quarter
    if ((warp >= 4 && warp < 4 + 4 * MOVERS) || (AD && warp == 0)) {
        const bool have = mbar_wait(&S.done, 0, a.status, DEV_TIMEOUT_MMA, &S.abort) && !*(volatile int *)&S.abort;
        tc_fence_after();
        // the features' warps take every MOVERS-th chunk of 16 columns (rows of the pass); warp 0 the adapter's
        const bool ad = AD && warp == 0;
        const int row = ad ? lane : (warp & 3) * 32 + lane, width = ad ? ru : TILE_ROWS, first = ad ? 0 : (warp - 4) >> 2;
        const uint32_t col = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (ad ? (uint32_t)a.bn : 0u);
        float *local = ad ? part_u : part;
        const uint32_t remote = ad ? pu : pa;
        const bool mine = !ad || lane < ru;
#pragma unroll 1
        for (int c0 = first * 16; have && c0 < M; c0 += ad ? 16 : 16 * MOVERS) {
            uint32_t v[16];
            tmem_ld_16cols(col + (uint32_t)c0, v);
            tmem_ld_wait();
            if (push) {
                int to = c0 % w.ks, at = slice * rpo + c0 / w.ks;  // destination CTA and row there
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    if (c0 + j >= M) break;
                    if (mine) st_cluster(map_cta(remote + (uint32_t)(at * width + row) * 4u, to), __uint_as_float(v[j]));
                    if (++to == w.ks) to = 0, ++at;
                }
            } else {
#pragma unroll
                for (int j = 0; j < 16; ++j)
                    if (c0 + j < M && mine) local[(c0 + j) * width + row] = __uint_as_float(v[j]);
            }
        }
        tc_fence_before();
    }
    __syncwarp();
    cluster_sync();
    if (warp == 0) tmem_dealloc(tmem, w.tmem_cols);

    // ---- rows slice, slice + slices, ...: one warp per row
    const uint32_t st4 = (uint32_t)(rpo * TILE_ROWS) * 4u, stu = (uint32_t)(rpo * ru) * 4u;  // slice strides (PUSH)
    float gn[4] = {0.f, 0.f, 0.f, 0.f};  // QK-norm gain of the lane's four features
    constexpr int LPH = DH / 4;          // lanes per head
    const int e0 = 4 * (lane % LPH);
    if (LIN == 0 && kind < 2) {
        const uint2 raw = __ldg(reinterpret_cast<const uint2 *>((kind == 0 ? w.q_norm : w.k_norm) + e0));
        const float2 x = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&raw.x));
        const float2 y = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&raw.y));
        gn[0] = x.x, gn[1] = x.y, gn[2] = y.x, gn[3] = y.y;
    }
    for (int m = slice + warp * w.ks; m < M; m += w.ks * (NT / 32)) {
        const int at = push ? m / w.ks : m;
        float lu = 0.f;  // lane i: the row's adapter intermediate u_i (gate|up: gate's, then up's)
        if (AD) lu = rbf(sum_slices(pu + (uint32_t)(at * ru + (lane < ru ? lane : 0)) * 4u, w.ks, stu, push));
        const float *bt = reinterpret_cast<const float *>(S.bt);
        if constexpr (LIN == 2) {
            // gate rows 2l, 2l + 1 and up rows 64 + 2l, 64 + 2l + 1 -> act features 64 tile + 2l, + 2l + 1
            float g[2], up[2];
            {
                float2 gs = make_float2(0.f, 0.f), us = gs;
                const uint32_t ga = pa + (uint32_t)(at * TILE_ROWS + 2 * lane) * 4u;
                for (int s = 0; s < w.ks; ++s) {
                    const uint32_t p = push ? ga + (uint32_t)s * st4 : map_cta(ga, s);
                    const float2 x = push ? ld_shared_v2(p) : ld_cluster_v2(p), y = push ? ld_shared_v2(p + 256u) : ld_cluster_v2(p + 256u);
                    gs = s == 0 ? x : make_float2(__fadd_rn(gs.x, x.x), __fadd_rn(gs.y, x.y));
                    us = s == 0 ? y : make_float2(__fadd_rn(us.x, y.x), __fadd_rn(us.y, y.y));
                }
                g[0] = gs.x, g[1] = gs.y, up[0] = us.x, up[1] = us.y;
            }
            if (AD) {
                float y[4] = {g[0], g[1], up[0], up[1]};
                add_delta(y, lu, lu, r, bt, 2 * lane, 64 + 2 * lane, r, dm.lora_scale);
                g[0] = y[0], g[1] = y[1], up[0] = y[2], up[1] = y[3];
            }
            float o[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                const float gt = rbf(g[e]);
                o[e] = __fmul_rn(__fdiv_rn(gt, __fadd_rn(1.0f, expf(-gt))), rbf(up[e]));
            }
            *reinterpret_cast<uint32_t *>(a.act + (size_t)m * dm.I + tile * 64 + 2 * lane) = pack_bf162(o[0], o[1]);
        } else {
            uint2 hraw = h1;
            uint2 *hp = reinterpret_cast<uint2 *>(a.h + (size_t)m * dm.H + ft) + lane;
            if ((LIN == 1 || LIN == 3) && m != m_first) hraw = __ldcg(hp);
            const float4 y4 = sum_slices4(pa + (uint32_t)(at * TILE_ROWS + 4 * lane) * 4u, w.ks, st4, push);
            float y[4] = {y4.x, y4.y, y4.z, y4.w};
            if (AD) add_delta(y, lu, lu, 0, bt, 4 * lane, 4 * lane + 2, r, dm.lora_scale);
#pragma unroll
            for (int e = 0; e < 4; ++e) y[e] = rbf(y[e]);
            if constexpr (LIN == 0) {
                const int pos = m == m_first ? pos1 : row_pos(m);
                const int page = kind == 0 ? 0 : (m == m_first ? page1 : row_page(m, pos));
                const int head = (ft - (kind == 0 ? 0 : (kind == 1 ? qw : qw + kvw))) / DH + lane / LPH;
                bool bad = page < 0;
                if (kind < 2) {
                    bad = bad || pos >= a.rope_rows;
                    float ssq = __fmul_rn(y[0], y[0]);
#pragma unroll
                    for (int j = 1; j < 4; ++j) ssq = __fadd_rn(ssq, __fmul_rn(y[j], y[j]));
#pragma unroll
                    for (int off = LPH / 2; off >= 1; off >>= 1) ssq = __fadd_rn(ssq, __shfl_xor_sync(0xffffffffu, ssq, off));
                    const float rs = rms_scale(ssq, DH, dm.eps);
                    float4 rope[2] = {rope1[0], rope1[1]};
                    if (m != m_first) row_rope(pos, rope);
                    const float4 ca = rope[0], cb = rope[1];
                    const float cs[4] = {ca.x, ca.z, cb.x, cb.z}, sn[4] = {ca.y, ca.w, cb.y, cb.w};
#pragma unroll
                    for (int j = 0; j < 4; ++j) y[j] = rbf(__fmul_rn(gn[j], rbf(__fmul_rn(y[j], rs))));
                    float z[4];
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        const float partner = __shfl_xor_sync(0xffffffffu, y[j], LPH / 2);
                        z[j] = e0 < DH / 2 ? __fsub_rn(__fmul_rn(y[j], cs[j]), __fmul_rn(partner, sn[j]))
                                           : __fadd_rn(__fmul_rn(y[j], cs[j]), __fmul_rn(partner, sn[j]));
                    }
#pragma unroll
                    for (int j = 0; j < 4; ++j) y[j] = z[j];
                }
                if (bad) {
                    latch_error(a.status, DEV_BAD_POSITION);
                    continue;
                }
                bf16 *dst = a.q + ((size_t)m * dm.Hq + head) * DH + e0;
                if (kind > 0)
                    dst = static_cast<bf16 *>(kind == 1 ? a.kv.k : a.kv.v) +
                          ((((size_t)w.layer * a.kv.n_pages + page) * dm.Hkv + head) * PAGE + (pos % PAGE)) * DH + e0;
                *reinterpret_cast<uint2 *>(dst) = make_uint2(pack_bf162(y[0], y[1]), pack_bf162(y[2], y[3]));
            } else {
                const __nv_bfloat162 *h2 = reinterpret_cast<const __nv_bfloat162 *>(&hraw);
                const float2 ha = __bfloat1622float2(h2[0]), hb = __bfloat1622float2(h2[1]);
                const float v[4] = {rbf(__fadd_rn(ha.x, y[0])), rbf(__fadd_rn(ha.y, y[1])), rbf(__fadd_rn(hb.x, y[2])),
                                    rbf(__fadd_rn(hb.y, y[3]))};
                *hp = make_uint2(pack_bf162(v[0], v[1]), pack_bf162(v[2], v[3]));
                float sq = __fmul_rn(v[0], v[0]);
#pragma unroll
                for (int e = 1; e < 4; ++e) sq = __fadd_rn(sq, __fmul_rn(v[e], v[e]));
#pragma unroll
                for (int off = 16; off >= 1; off >>= 1) sq = __fadd_rn(sq, __shfl_xor_sync(0xffffffffu, sq, off));
                if (lane == 0) a.ss[(size_t)m * (dm.H / TILE_ROWS) + tile] = sq;
            }
        }
    }
    if (!push) cluster_sync();  // no CTA leaves while another still reads its partials
}

// ------------------------------------------------------------------ attention step
//
// Grid (splits, KV heads, sequences): a CTA takes one 128-key split of a (sequence, KV head); units of one
// 16-row query tile against the split (or a 64-key half of it) go to the warps, as in attn_split
// (pass_kernel.cu), and each leaves a partial result (m, l, O) per row.
//
// CLUSTER: the group's CTAs are a cluster (a power of two of them, so some may have no split).  A row's
// partial results go straight to the shared memory of CTA row % CTAs, which merges them in key order
// after the cluster barrier.  Otherwise (more splits than a portable cluster has CTAs, or more groups
// than the GPU holds clusters of: then clusters wait for one another's SMs) they go to memory and
// k_step_merge merges them.
//
// A step of ~6.5 us is bound by its warps' latency, not by K/V bytes (17 rows at 512 tokens: scores, softmax and PV
// 2.4 us, exchange 1.4, merge 1.3).  The q rows lie in shared memory and each MMA group's fragments are
// loaded before its MMAs; with all of q's fragments in registers the compiler had too few left to batch
// those loads (verify pass 779 us against 769; 4096 tokens 934 against 899).
constexpr int SA_WARPS = 6;   // compute warps of a cluster's CTA: the units of 17 rows with two heads a group
// compute warps of a single split's CTA, compiled for three CTAs an SM: one-row passes have three there, 17 rows two
// (their q rows take shared memory), and the fewer registers suit both (17 rows at 4096 tokens, us a layer of a verify
// pass: 33.1; compiled for two 34.4)
constexpr int SG_WARPS = 4;
constexpr int SA_STATS = 4;   // partial results per row at most: 32 x this

// Merge of one row's nv partial results in key order, relative to the row's overall maximum (attn_combine in
// pass_kernel.cu): lane l gathers the statistics of partials l, l + 32, ... and the outputs 4l..4l+3.
template <int DH, typename FS, typename FO>
__device__ __forceinline__ void merge_row(int nv, int lane, FS stat, FO out, bf16 *dst) {
    constexpr int OB = 8;  // partial outputs in flight
    const int c = lane < DH / 4 ? 4 * lane : 0;
    float2 st[SA_STATS];
    float4 o[OB];
    float mx = -INFINITY;
#pragma unroll
    for (int i = 0; i < SA_STATS; ++i) st[i] = 32 * i + lane < nv ? stat(32 * i + lane) : make_float2(-INFINITY, 0.f);
#pragma unroll
    for (int u = 0; u < OB; ++u) o[u] = out(min(u, nv - 1), c);
#pragma unroll
    for (int i = 0; i < SA_STATS; ++i)
        if (st[i].y > 0.f) mx = fmaxf(mx, st[i].x);
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    float4 num = make_float4(0.f, 0.f, 0.f, 0.f);
    float den = 0.f;
#pragma unroll
    for (int i = 0; i < SA_STATS; ++i) {
        if (32 * i >= nv) break;
        const float wl = __expf(st[i].x - mx);
#pragma unroll 1
        for (int p0 = 32 * i; p0 < min(nv, 32 * i + 32); p0 += OB) {
            if (p0 > 0)
#pragma unroll
                for (int u = 0; u < OB; ++u) o[u] = out(min(p0 + u, nv - 1), c);
#pragma unroll
            for (int u = 0; u < OB; ++u) {
                if (p0 + u >= nv) break;
                const float wt = __shfl_sync(0xffffffffu, wl, (p0 + u) & 31);
                const float l = __shfl_sync(0xffffffffu, st[i].y, (p0 + u) & 31);
                if (!(l > 0.f)) continue;  // the row saw no key in this partial result
                den = __fadd_rn(den, __fmul_rn(wt, l));
                num = make_float4(__fadd_rn(num.x, __fmul_rn(wt, o[u].x)), __fadd_rn(num.y, __fmul_rn(wt, o[u].y)),
                                  __fadd_rn(num.z, __fmul_rn(wt, o[u].z)), __fadd_rn(num.w, __fmul_rn(wt, o[u].w)));
            }
        }
    }
    if (lane < DH / 4)
        *reinterpret_cast<uint2 *>(dst + 4 * lane) = make_uint2(pack_bf162(__fdiv_rn(num.x, den), __fdiv_rn(num.y, den)),
                                                                pack_bf162(__fdiv_rn(num.z, den), __fdiv_rn(num.w, den)));
}

template <int DH, bool BLK, bool CLUSTER>
__global__ void __launch_bounds__(32 * (CLUSTER ? SA_WARPS : SG_WARPS) + 32, CLUSTER ? 1 : 3)
    k_step_attn(const __grid_constant__ CUtensorMap kmap, const __grid_constant__ CUtensorMap vmap,
                const __grid_constant__ StepArgs a, int layer, int parts, const __grid_constant__ StepSplits sp) {
    constexpr int WARPS = CLUSTER ? SA_WARPS : SG_WARPS, PITCH = DH + 4, QP = ATT_Q_PITCH(DH);
    constexpr int DT = DH / 8, SUBS = DH / 64, NP = ATT_SPLIT / PAGE;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ uint64_t full;
    const Dims &dm = a.dm;
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    // (without clusters the sequences' splits lie end to end along x)
    int bl = blockIdx.z;
    if (!CLUSTER)
        while (blockIdx.x >= sp.start[bl + 1]) ++bl;
    const int split = blockIdx.x - (CLUSTER ? 0 : sp.start[bl]), cs = gridDim.x, g = blockIdx.y;
    const int b = a.pd.b0 + bl, R = a.pd.R, grp = dm.Hq / dm.Hkv, RH = R * grp;
    const int sub_sh = a.att_subs - 1, HALF = ATT_SPLIT >> sub_sh;  // one or two partial results per split
    // CLUSTER: the partial results of the rows that this CTA merges
    const int cs_sh = __ffs(cs) - 1, rpo = (RH + cs - 1) / cs;           // (cs is a power of two there)
    const uint32_t sq = smem_u32(base + 2 * SUBS * ATT_SUB_BYTES);       // q rows (16 a tile), QP bytes each
    const uint32_t po = sq + (uint32_t)((RH + 15) / 16 * 16 * QP);       // [parts][rpo][PITCH]
    const uint32_t pml = po + (uint32_t)(parts * rpo * PITCH) * 4u;      // [parts][rpo] (m, l)
    if (threadIdx.x == 0) {
        mbar_init(&full, 1);
        fence_mbarrier_init();
        prefetch_tensormap(&kmap);
        prefetch_tensormap(&vmap);
    }
    __syncthreads();
    if (CLUSTER) cluster_arrive();  // (this CTA's shared memory exists: its peers wait for that before they write there)
    pdl_launch();
    // the cached length was set by a kernel that finished before this pass began
    const int L = a.L[b], T = L + R, nsp = (T + ATT_SPLIT - 1) / ATT_SPLIT, k0 = split * ATT_SPLIT;
    const bool active = split < nsp;

    if (warp == WARPS) {
        // ---- producer warp: lane p the page p of the split.  Pages entirely below L hold earlier passes' keys and
        // are requested at once; the block's own after the wait.
        if (active) {
            const int pg = split * NP + lane, kp = k0 + lane * PAGE;
            const int page = lane < NP && kp < T && pg < a.kv.pages_per_seq ? a.kv.page_table[(size_t)b * a.kv.pages_per_seq + pg] : -1;
            auto request = [&](bool cached) {
                const unsigned mask = __ballot_sync(0xffffffffu, page >= 0 && (kp + PAGE <= L) == cached);
                const uint32_t bytes = (uint32_t)__popc(mask) * 2u * SUBS * PAGE * 128u;
                if (lane == 0) {
                    if (!cached)
                        mbar_arrive_expect_tx(&full, bytes);
                    else if (bytes)
                        mbar_expect_tx(&full, bytes);
                }
                __syncwarp();
#pragma unroll 1
                for (int c0 = 0; c0 < NP * 2 * SUBS; c0 += 32) {
                    const int cp = c0 + lane, p = cp / (2 * SUBS), q = cp % (2 * SUBS);
                    const int phys = __shfl_sync(0xffffffffu, page, p & 31);
                    if (p < NP && ((mask >> p) & 1u))
                        tma_load_2d(base + q * ATT_SUB_BYTES + p * PAGE * 128, q / SUBS ? &vmap : &kmap, (q % SUBS) * 64,
                                    ((layer * a.kv.n_pages + phys) * dm.Hkv + g) * PAGE, &full);
                }
            };
            request(true);
            pdl_wait();
            fence_proxy_async_global();
            request(false);
            mbar_wait(&full, 0, nullptr, 0, nullptr);  // (the copies land before this CTA's memory goes)
        }
        if (CLUSTER) cluster_wait();
    } else {
        const int gq = lane >> 2, tq = lane & 3, n_units = ((RH + 15) / 16) << sub_sh;
        const float scale = a.att_scale;
        const uint32_t ka = smem_u32(base) + attn_k_lane(lane);
        const uint32_t va = smem_u32(base + SUBS * ATT_SUB_BYTES) + attn_v_lane(lane), qoff = attn_q_lane<DH>(lane);
        pdl_wait();
        // the group's q rows through L2 while the block's pages land
        if (active) {
            for (int q = threadIdx.x; q < RH * (DH / 8); q += 32 * WARPS) {
                const int qv = q / (DH / 8), c = q % (DH / 8);
                cp_async16_at(sq + (uint32_t)(qv * QP + c * 16),
                              a.q + ((size_t)(bl * R + qv / grp) * dm.Hq + g * grp + qv % grp) * DH + c * 8);
            }
            cp_async_commit();
            cp_async_wait_all();
            asm volatile("bar.sync 1, %0;" ::"n"(32 * WARPS) : "memory");
        }
        if (CLUSTER) cluster_wait();
        bool landed = false;
#pragma unroll 1
        for (int unit = warp; active && unit < n_units; unit += WARPS) {
            const int half = unit & sub_sh, mt = unit >> sub_sh, kb = half * HALF;
            const int qv0 = mt * 16 + gq, qv1 = qv0 + 8;
            const bool val0 = qv0 < RH, val1 = qv1 < RH;
            const int i0 = val0 ? qv0 / grp : 0, i1 = val1 ? qv1 / grp : 0;
            if (!landed && !(landed = mbar_wait(&full, 0, a.status, DEV_TIMEOUT_LOAD, nullptr))) break;
            // last visible key of each row (the draft's mask rows see the whole block)
            const int lim0 = val0 ? ((BLK && i0 >= 1) ? T - 1 : L + i0) : -1;
            const int lim1 = val1 ? ((BLK && i1 >= 1) ? T - 1 : L + i1) : -1;
            float m0 = -INFINITY, m1 = -INFINITY, l0 = 0.f, l1 = 0.f;
            float oc[DT][4];
#pragma unroll
            for (int dt = 0; dt < DT; ++dt) oc[dt][0] = oc[dt][1] = oc[dt][2] = oc[dt][3] = 0.f;
            const int kend = min(HALF, T - (k0 + kb));
#pragma unroll 1
            for (int c0 = 0; c0 < kend; c0 += 32) {
                float sc[4][4];
                attn_scores_sq<DH>(ka + (kb + c0) * 128, sq + (uint32_t)(mt * 16 * QP) + qoff, sc);
                float c0m = -INFINITY, c1m = -INFINITY;
#pragma unroll
                for (int nt = 0; nt < 4; ++nt)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int kp = k0 + kb + c0 + nt * 8 + 2 * tq + e;
                        sc[nt][e] = kp <= lim0 ? __fmul_rn(sc[nt][e], scale) : -INFINITY;
                        sc[nt][2 + e] = kp <= lim1 ? __fmul_rn(sc[nt][2 + e], scale) : -INFINITY;
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
                    // V of keys at or past T is zero in the fragments (see attn_split)
                    const int kst = k0 + kb + c0 + kstep * 16;
                    uint32_t ma = 0xFFFFFFFFu, mb = 0xFFFFFFFFu;
                    if (kst + 16 > T) {
                        const int kf = kst + 2 * tq;
                        ma = (kf < T ? 0x0000FFFFu : 0u) | (kf + 1 < T ? 0xFFFF0000u : 0u);
                        mb = (kf + 8 < T ? 0x0000FFFFu : 0u) | (kf + 9 < T ? 0xFFFF0000u : 0u);
                    }
                    attn_pv<DH>(va + (kb + c0 + kstep * 16) * 128, pa, ma, mb, oc);
                }
            }
            l0 += __shfl_xor_sync(0xffffffffu, l0, 1);
            l0 += __shfl_xor_sync(0xffffffffu, l0, 2);
            l1 += __shfl_xor_sync(0xffffffffu, l1, 1);
            l1 += __shfl_xor_sync(0xffffffffu, l1, 2);
            const int part = (split << sub_sh) + half;
            auto store = [&](bool val, int qv, int i, float m, float l, int e) {
                if (!val) return;
                if constexpr (CLUSTER) {
                    const int row = part * rpo + (qv >> cs_sh), to = qv & (cs - 1);
                    const uint32_t dst = map_cta(po + (uint32_t)(row * PITCH + 2 * tq) * 4u, to);
                    if (tq == 0) st_cluster_v2(map_cta(pml + (uint32_t)row * 8u, to), m, l);
#pragma unroll
                    for (int dt = 0; dt < DT; ++dt) st_cluster_v2(dst + dt * 32, oc[dt][e], oc[dt][e + 1]);
                } else {
                    const size_t row = ((size_t)(bl * R + i) * dm.Hq + g * grp + qv % grp) * a.att_splits_alloc + part;
                    float *dst = a.o_part + row * DH + 2 * tq;
                    if (tq == 0) a.ml_part[row] = make_float2(m, l);
#pragma unroll
                    for (int dt = 0; dt < DT; ++dt) *reinterpret_cast<float2 *>(dst + dt * 8) = make_float2(oc[dt][e], oc[dt][e + 1]);
                }
            };
            store(val0, qv0, i0, m0, l0, 0);
            store(val1, qv1, i1, m1, l1, 2);
        }
    }
    if constexpr (CLUSTER) {
        __syncwarp();
        cluster_sync();
        if (warp < SA_WARPS)
            for (int qv = split + warp * cs; qv < RH; qv += cs * SA_WARPS)
                merge_row<DH>(
                    nsp << sub_sh, lane, [&](int p) { return ld_shared_v2(pml + (uint32_t)(p * rpo + (qv >> cs_sh)) * 8u); },
                    [&](int p, int c) { return ld_shared_v4(po + (uint32_t)((p * rpo + (qv >> cs_sh)) * PITCH + c) * 4u); },
                    a.attn + ((size_t)(bl * R + qv / grp) * dm.Hq + g * grp + qv % grp) * DH);
    }
}

// Merge of the partial results in memory (as merge_row): a block per (row, query head), a thread per
// dimension, so that up to 32 partial outputs are on their way at once.
template <int DH>
__global__ void __launch_bounds__(DH) k_step_merge(const __grid_constant__ StepArgs a) {
    constexpr int OB = 32;
    const int lane = threadIdx.x & 31, m = blockIdx.x / a.dm.Hq;
    pdl_launch();
    const int nv = (a.L[a.pd.b0 + m / a.pd.R] + a.pd.R + ATT_SPLIT - 1) / ATT_SPLIT * a.att_subs;
    const size_t row = (size_t)blockIdx.x * a.att_splits_alloc;
    const float *op = a.o_part + row * DH + threadIdx.x;
    pdl_wait();
    float2 st[SA_STATS];
    float o[OB];
#pragma unroll
    for (int i = 0; i < SA_STATS; ++i)
        st[i] = 32 * i + lane < nv ? __ldcg(a.ml_part + row + 32 * i + lane) : make_float2(-INFINITY, 0.f);
#pragma unroll
    for (int u = 0; u < OB; ++u) o[u] = u < nv ? __ldcg(op + (size_t)u * DH) : 0.f;
    float mx = -INFINITY;
#pragma unroll
    for (int i = 0; i < SA_STATS; ++i)
        if (st[i].y > 0.f) mx = fmaxf(mx, st[i].x);
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    float num = 0.f, den = 0.f;
#pragma unroll
    for (int i = 0; i < SA_STATS; ++i) {
        if (32 * i >= nv) break;
        if (i > 0)
#pragma unroll
            for (int u = 0; u < OB; ++u) o[u] = 32 * i + u < nv ? __ldcg(op + (size_t)(32 * i + u) * DH) : 0.f;
        const float wl = __expf(st[i].x - mx);
#pragma unroll
        for (int u = 0; u < OB; ++u) {
            if (32 * i + u >= nv) break;
            const float wt = __shfl_sync(0xffffffffu, wl, u), l = __shfl_sync(0xffffffffu, st[i].y, u);
            if (!(l > 0.f)) continue;  // the row saw no key in this partial result
            den = __fadd_rn(den, __fmul_rn(wt, l));
            num = __fadd_rn(num, __fmul_rn(wt, o[u]));
        }
    }
    a.attn[(size_t)blockIdx.x * DH + threadIdx.x] = f2bf(__fdiv_rn(num, den));
}

// ------------------------------------------------------------------ ends of the pass

// One warp per row and 128-feature tile: token or mask embedding -> h and the tile's sum of squares (as
// do_embed in pass_kernel.cu).
__global__ void __launch_bounds__(256) k_step_embed(const __grid_constant__ StepArgs a, const bf16 *__restrict__ embed_tiled,
                                                    const bf16 *__restrict__ mask_embed) {
    const int lane = threadIdx.x & 31, H = a.dm.H, nt = H / TILE_ROWS;
    const int un = blockIdx.x * 8 + (threadIdx.x >> 5);
    pdl_begin();
    if (un >= a.pd.M * nt) return;
    const int m = un / nt, t = un % nt;
    int tok = a.ids[m];
    if (tok >= a.dm.V || tok < -1 || (tok == -1 && !a.pd.adapter)) {
        if (lane == 0) latch_error(a.status, DEV_BAD_TOKEN);
        tok = 0;
    }
    float s = 0.f;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int f = t * TILE_ROWS + lane + 32 * e;
        const bf16 v = tok >= 0 ? *tiled_at(embed_tiled, H, tok, f) : mask_embed[f];
        a.h[(size_t)m * H + f] = v;
        const float x = bf2f(v);
        s = e == 0 ? __fmul_rn(x, x) : __fadd_rn(s, __fmul_rn(x, x));
    }
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) s = __fadd_rn(s, __shfl_xor_sync(0xffffffffu, s, off));
    if (lane == 0) a.ss[(size_t)m * nt + t] = s;
}

// final RMSNorm of the read-out rows, one warp per row
__global__ void __launch_bounds__(256) k_step_final(const __grid_constant__ StepArgs a, const bf16 *__restrict__ gain, bf16 *x_ro) {
    const int lane = threadIdx.x & 31, H = a.dm.H, nt = H / TILE_ROWS;
    const int ro = blockIdx.x * 8 + (threadIdx.x >> 5);
    pdl_begin();
    if (ro >= a.pd.nb * a.pd.ro_count) return;
    const int m = ro / a.pd.ro_count * a.pd.R + a.pd.ro_first + ro % a.pd.ro_count;
    float sum = 0.f;
    for (int t = 0; t < nt; ++t) {
        const float v = __ldcg(a.ss + (size_t)m * nt + t);
        sum = t == 0 ? v : __fadd_rn(sum, v);
    }
    const float rs = rms_scale(sum, H, a.dm.eps);
    for (int c = lane; c < H / 8; c += 32) {
        uint4 hv = __ldcg(reinterpret_cast<const uint4 *>(a.h + (size_t)m * H) + c);
        const uint4 gv = __ldg(reinterpret_cast<const uint4 *>(gain) + c);
        __nv_bfloat162 *h2 = reinterpret_cast<__nv_bfloat162 *>(&hv);
        const __nv_bfloat162 *g2 = reinterpret_cast<const __nv_bfloat162 *>(&gv);
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const float2 f = __bfloat1622float2(h2[e]);
            h2[e] = __hmul2(g2[e], __floats2bfloat162_rn(__fmul_rn(f.x, rs), __fmul_rn(f.y, rs)));
        }
        reinterpret_cast<uint4 *>(x_ro + (size_t)ro * H)[c] = hv;
    }
}

// ------------------------------------------------------------------ host side

constexpr int ST_SMEM = 216 * 1024;   // dynamic shared memory of one CTA at most
constexpr int ST_MAX_CLUSTER = 16;
// Rows up to which partial sums are pushed: a pushed row costs a scalar remote store per thread (~40 ns), pulling
// costs a remote round trip and a second cluster barrier (~0.8 us) once (17 rows: verify pass 896 us pulled, 799
// pushed; 136 rows: 1823 pulled, 2032 pushed).  Between them, us a layer, verify / draft: 33 rows 36.3 / 44.5
// pulled, 35.1 / 44.2 pushed; 48 rows 40.2 / 47.9 and 39.0 / 48.7; 64 rows 46.7 / 55.4 and 45.4 / 56.7.
constexpr int ST_PUSH_ROWS = 32;

static int step_bn(int M) { return std::max(32, (M + 15) / 16 * 16); }

// Ring atoms of a linear with katoms per slice (0: does not fit), whether its partial sums have room behind the
// ring (push), and the dynamic shared memory.
static int lin_ring(int bn, int M, int katoms, int ks, bool ad, int ru, int *push, size_t *smem) {
    for (int ra : {katoms, ST_HALF}) {
        const int ring = ra * (TILE_BYTES + (ad ? ST_A_BYTES : 0) + bn * 128);
        const int behind = (int)sizeof(float) * ks * ((M + ks - 1) / ks) * (TILE_ROWS + ru);
        if (ring + 1024 > ST_SMEM) continue;
        *push = M <= ST_PUSH_ROWS && ring + behind + 1024 <= ST_SMEM ? 1 : 0;
        *smem = (size_t)ring + (*push ? behind : 0) + 1024;
        if (*push || (int)sizeof(float) * M * (TILE_ROWS + ru) <= ring) return ra;
    }
    return 0;
}

static int attn_smem(const Dims &dm, int R, int parts, int rows) {
    return 2 * (dm.d / 64) * ATT_SUB_BYTES + (R * (dm.Hq / dm.Hkv) + 15) / 16 * 16 * ATT_Q_PITCH(dm.d) + parts * rows * ((dm.d + 4) * 4 + 8) + 1024;
}

// The attention's form: the CTAs of a cluster per (sequence, KV head), a split each, or 0: one CTA per split and
// a merge kernel.  Clusters while a portable one has a CTA for each split, the partial results of the rows
// that a CTA merges fit, and every cluster has its SMs at once.
static int attn_cluster(const Dims &dm, const PassDesc &pd, int subs, int nsplit, size_t *smem) {
    int c = 1;
    while (c < nsplit && c < 8) c *= 2;
    *smem = attn_smem(dm, pd.R, nsplit * subs, (pd.R * (dm.Hq / dm.Hkv) + c - 1) / c);
    return c >= nsplit && pd.nb * dm.Hkv * c <= gemm_ctas() && *smem <= (size_t)ST_SMEM ? c : 0;
}

// Slices of a linear at most: one cluster, and one that the device can place (0.6B shape but the hidden size, us a layer
// of a verify pass, persistent kernel in brackets: 12 slices 57 (85), 13 64 (118), 14 72 (109), 15 93 (131), 16 76
// (114); a draft 93 (102), 138 (138), 116 (130), 159 (157), 126 (137)).
static int max_slices() {
    static const int n = largest_cluster((const void *)k_step_linear<0, true, 128, 512>, 512, ST_SMEM, ST_MAX_CLUSTER);
    return n;
}

bool step_pass_fits(const Dims &dm, const PassDesc &pd, int subs, int nsplit) {
    const int K[4] = {dm.H, dm.Hq * dm.d, dm.H, dm.I};
    const int bn = step_bn(pd.M);
    if (pd.M > 256 || dm.r > ST_RANK) return false;
    for (int lin = 0; lin < 4; ++lin) {
        const int ka = mk_slice_atoms(lin, K[lin]);
        const int ks = K[lin] / (ka * KT), ru = pd.adapter ? (lin == 2 ? 2 : 1) * dm.r : 0;
        int push;
        size_t smem;
        if (ks > max_slices() || lin_ring(bn, pd.M, ka, ks, pd.adapter, ru, &push, &smem) == 0) return false;
    }
    // (statistics a merging warp holds; a split's pages and the group's q rows)
    return nsplit * subs <= 32 * SA_STATS && attn_smem(dm, pd.R, 0, 0) <= ST_SMEM;
}

template <typename... P, typename... A>
static cudaError_t launch_step(void (*kernel)(P...), dim3 grid, dim3 cluster, int threads, size_t smem, cudaStream_t st,
                               A &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3((unsigned)threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = cluster.x;
    attr[1].val.clusterDim.y = cluster.y;
    attr[1].val.clusterDim.z = cluster.z;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// More threads for more rows: staging and finishing rows are loops over them (136 rows, 0.6B
// shape: verify pass 1763 us with 256 threads, 1619 with 512; at 17 rows the wider CTA starts later).  The line is
// higher than it need be: us a layer, verify / draft, with 256 and with 512 threads: 33 rows 36.3 / 44.5 and
// 34.4 / 42.2, 64 rows 46.7 / 55.4 and 42.6 / 52.3, 68 rows 41.2 / 53.9 and 38.8 / 50.2.
static int lin_threads(int M) { return M <= 64 ? 256 : 512; }

template <int DH, int NT>
static cudaError_t launch_lin(int lin, bool ad, dim3 grid, size_t smem, const StepArgs &a, const StepLin &w, cudaStream_t st) {
    const dim3 cl(1, grid.y);
#define STEP_LIN(L)                                                                                              \
    return ad ? launch_step(k_step_linear<L, true, DH, NT>, grid, cl, NT, smem, st, a, w)                        \
              : launch_step(k_step_linear<L, false, DH, NT>, grid, cl, NT, smem, st, a, w)
    switch (lin) {
        case 0: STEP_LIN(0);
        case 1: STEP_LIN(1);
        case 2: STEP_LIN(2);
        default: STEP_LIN(3);
    }
#undef STEP_LIN
}

cudaError_t launch_step_linear(int lin, StepArgs &a, StepLin &w, cudaStream_t st) {
    const bool ad = a.pd.adapter != 0;
    a.bn = step_bn(a.pd.M);
    w.k_tiles = w.K / KT;
    w.katoms = mk_slice_atoms(lin, w.K);
    w.ks = w.k_tiles / w.katoms;
    size_t smem = 0;
    w.ring_atoms = lin_ring(a.bn, a.pd.M, w.katoms, w.ks, ad, ad ? (lin == 2 ? 2 : 1) * a.dm.r : 0, &w.push, &smem);
    if (w.ring_atoms == 0 || w.ks > ST_MAX_CLUSTER) return cudaErrorInvalidValue;
    w.tmem_cols = 32;
    while ((int)w.tmem_cols < (ad ? 2 : 1) * a.bn) w.tmem_cols <<= 1;
    if (lin == 1 || lin == 3)
        if (!encode_bf16_map(&w.xmap, lin == 1 ? (const void *)a.attn : (const void *)a.act, a.rows_alloc, w.K,
                             w.short_x ? a.bn - 16 : a.bn))
            return cudaErrorInvalidValue;
    const dim3 grid(w.n_main / TILE_ROWS, w.ks);
    if (lin_threads(a.pd.M) == 256)
        return a.dm.d == 128 ? launch_lin<128, 256>(lin, ad, grid, smem, a, w, st) : launch_lin<64, 256>(lin, ad, grid, smem, a, w, st);
    return a.dm.d == 128 ? launch_lin<128, 512>(lin, ad, grid, smem, a, w, st) : launch_lin<64, 512>(lin, ad, grid, smem, a, w, st);
}

template <int DH, bool BLK>
static cudaError_t launch_attn(const StepArgs &a, const CUtensorMap &kmap, const CUtensorMap &vmap, int layer,
                               const StepSplits &sp, cudaStream_t st) {
    int nsplit = 0;
    for (int b = 0; b < a.pd.nb; ++b) nsplit = std::max(nsplit, sp.start[b + 1] - sp.start[b]);
    size_t smem;
    const int cs = attn_cluster(a.dm, a.pd, a.att_subs, nsplit, &smem);
    if (cs > 0)
        return launch_step(k_step_attn<DH, BLK, true>, dim3(cs, a.dm.Hkv, a.pd.nb), dim3(cs), 32 * SA_WARPS + 32, smem, st,
                           kmap, vmap, a, layer, nsplit * a.att_subs, sp);
    cudaError_t e = launch_step(k_step_attn<DH, BLK, false>, dim3(sp.start[a.pd.nb], a.dm.Hkv), dim3(1), 32 * SG_WARPS + 32,
                                attn_smem(a.dm, a.pd.R, 0, 0), st, kmap, vmap, a, layer, 0, sp);
    if (e != cudaSuccess) return e;
    return launch_pdl(k_step_merge<DH>, a.pd.M * a.dm.Hq, DH, 0, st, a);
}

cudaError_t launch_step_attn(const StepArgs &a, const CUtensorMap &kmap, const CUtensorMap &vmap, int layer,
                             const StepSplits &sp, cudaStream_t st) {
    const bool blk = a.pd.mask_mode == MASK_BLOCK_DRAFT;
    if (a.dm.d == 128)
        return blk ? launch_attn<128, true>(a, kmap, vmap, layer, sp, st) : launch_attn<128, false>(a, kmap, vmap, layer, sp, st);
    return blk ? launch_attn<64, true>(a, kmap, vmap, layer, sp, st) : launch_attn<64, false>(a, kmap, vmap, layer, sp, st);
}

cudaError_t launch_step_embed(const StepArgs &a, const void *embed_tiled, const void *mask_embed, cudaStream_t st) {
    return launch_pdl(k_step_embed, (a.pd.M * (a.dm.H / TILE_ROWS) + 7) / 8, 256, 0, st, a,
                      static_cast<const bf16 *>(embed_tiled), static_cast<const bf16 *>(mask_embed));
}

cudaError_t launch_step_final(const StepArgs &a, const void *gain, void *x_ro, cudaStream_t st) {
    return launch_pdl(k_step_final, (a.pd.nb * a.pd.ro_count + 7) / 8, 256, 0, st, a, static_cast<const bf16 *>(gain),
                      static_cast<bf16 *>(x_ro));
}

cudaError_t configure_step_kernels() {
    cudaError_t e = cudaSuccess;
    auto set = [&](const void *f) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, ST_SMEM);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
        // an SM changes its split of shared memory and L1 only when it is empty: with one split for all steps a
        // step's CTAs can start beside the one before
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    };
#define STEP_SET(L, NT)                                  \
    set((const void *)k_step_linear<L, true, 128, NT>);  \
    set((const void *)k_step_linear<L, false, 128, NT>); \
    set((const void *)k_step_linear<L, true, 64, NT>);   \
    set((const void *)k_step_linear<L, false, 64, NT>)
    STEP_SET(0, 256);
    STEP_SET(1, 256);
    STEP_SET(2, 256);
    STEP_SET(3, 256);
    STEP_SET(0, 512);
    STEP_SET(1, 512);
    STEP_SET(2, 512);
    STEP_SET(3, 512);
#undef STEP_SET
#define STEP_SET(DH, BLK)                            \
    set((const void *)k_step_attn<DH, BLK, true>);   \
    set((const void *)k_step_attn<DH, BLK, false>)
    STEP_SET(128, true);
    STEP_SET(128, false);
    STEP_SET(64, true);
    STEP_SET(64, false);
#undef STEP_SET
    for (const void *f : {(const void *)k_step_merge<128>, (const void *)k_step_merge<64>, (const void *)k_step_embed,
                          (const void *)k_step_final})
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
    return e;
}

}  // namespace pbd
