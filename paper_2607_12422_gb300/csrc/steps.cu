// steps.cu -- a decoding pass (draft, verify, plain decoding) as a chain of small dependent kernels.
//
// A layer is five kernels: q|k|v (+ QK-norm, RoPE, K/V write), attention, o (+ residual), gate|up (+ SiLU),
// down (+ residual).  Each is one step of the chain, bound by latency and not by its few megabytes of
// weights, so the design removes what the chain waits for:
//   - A linear's K slices (256 wide, gate|up 512) are one thread-block cluster per 128-feature tile.  The
//     slices' fp32 partial sums stay in shared memory; after a cluster barrier CTA s finishes rows s,
//     s + slices, ... reading its peers through distributed shared memory.  The attention's key
//     splits of a (sequence, KV head) are a cluster too, and merge the same way.  No partial sum or
//     completion counter goes through global memory.
//   - The kernels launch dependent: a CTA sets itself up and requests its weights (or the cached K/V
//     pages) while the step before it still runs, and waits only for its activations.
//
// The arithmetic is the persistent pass kernel's (pass_kernel.cu), operation for operation: K slices and
// their order, key partition, every sum and rounding.  That kernel remains for contexts limited to fewer
// CTAs than SMs and for shapes whose slices or partial results do not fit a cluster; rows.cu computes the
// same for prompts.
//
// 0.6B shape, all layers of one pass (the persistent kernel in brackets), us: verify 896 (1136), draft 1159
// (1287), one-row decoding 720 (945) at 512 tokens of context; 1057 (1430), 1281 (1579), 893 (1196) at 4096;
// 1823 (3637), 2424 (4080), 1025 (1778) for eight sequences of 420 to 1757 tokens.
#include <algorithm>
#include <cmath>

#include "attn.cuh"
#include "common.cuh"
#include "pbd_internal.h"

namespace pbd {

constexpr int ST_THREADS = 256;
constexpr int ST_STAGERS = 192;    // threads that stage a normalised operand (warps 2-7)
constexpr int ST_HALF = 4;         // 64-wide K atoms per half (256 of K)
constexpr int ST_RANK = 16;        // adapter rank (8 or 16)
constexpr int ST_A_BYTES = 2 * ST_RANK * 128;  // adapter rows of one K atom (gate and up: two ranks)

__device__ __forceinline__ uint32_t map_cta(uint32_t addr, int rank) {
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(addr), "r"(rank));
    return a;
}
__device__ __forceinline__ float4 ld_cluster_v4(uint32_t a) {
    float4 v;
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(a)
                 : "memory");
    return v;
}
__device__ __forceinline__ float2 ld_cluster_v2(uint32_t a) {
    float2 v;
    asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ float ld_cluster(uint32_t a) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void bar_stagers() { asm volatile("bar.sync 1, 192;" ::: "memory"); }

__device__ __forceinline__ float4 add4(float4 a, float4 b) {
    return make_float4(__fadd_rn(a.x, b.x), __fadd_rn(a.y, b.y), __fadd_rn(a.z, b.z), __fadd_rn(a.w, b.w));
}

// ------------------------------------------------------------------ linear step

struct StepLinState {
    uint64_t wfull[2], xfull[2], hdone, done;
    uint32_t tmem_slot;
    int abort;
    float rs[256];  // 1/rms of each row (normalised operands)
    // the adapter's B rows of the tile: row j at chunk j * (r / 8) + j / 4 (16 bytes of padding after
    // every four rows: a reducing lane reads rows 4l..4l+3)
    uint4 brows[TILE_ROWS * ST_RANK / 8 + TILE_ROWS / 4];
};

// sum over the slices of four features (float4) or of one adapter row, in slice order
__device__ __forceinline__ float4 sum_slices4(uint32_t a, int ks) {
    float4 y = ld_cluster_v4(map_cta(a, 0));
    for (int s0 = 1; s0 < ks; s0 += 4) {
        float4 v[4];
#pragma unroll
        for (int s = 0; s < 4; ++s) v[s] = ld_cluster_v4(map_cta(a, min(s0 + s, ks - 1)));
#pragma unroll
        for (int s = 0; s < 4; ++s)
            if (s0 + s < ks) y = add4(y, v[s]);
    }
    return y;
}
__device__ __forceinline__ float sum_slices(uint32_t a, int ks) {
    float y = ld_cluster(map_cta(a, 0));
    for (int s0 = 1; s0 < ks; s0 += 4) {
        float v[4];
#pragma unroll
        for (int s = 0; s < 4; ++s) v[s] = ld_cluster(map_cta(a, min(s0 + s, ks - 1)));
#pragma unroll
        for (int s = 0; s < 4; ++s)
            if (s0 + s < ks) y = __fadd_rn(y, v[s]);
    }
    return y;
}

// the adapter intermediates u_0 .. u_{r-1} of one row, from lanes base, base + 1, ...
__device__ __forceinline__ void spread_u(float lane_u, int base, float (&u)[ST_RANK]) {
#pragma unroll
    for (int j = 0; j < ST_RANK; ++j) u[j] = __shfl_sync(0xffffffffu, lane_u, base + j);
}
// u . B[j] over the rank, in order
__device__ __forceinline__ float lora_dot_s(const float (&u)[ST_RANK], const uint4 *brows, int j, int r) {
    float a = 0.f;
    const uint4 *b = brows + j * (r / 8) + (j >> 2);
#pragma unroll
    for (int q = 0; q < ST_RANK / 8; ++q) {
        if (q * 8 >= r) break;
        const uint4 w = b[q];
        const bf16 *e = reinterpret_cast<const bf16 *>(&w);
#pragma unroll
        for (int i = 0; i < 8; ++i) a = __fadd_rn(a, __fmul_rn(u[q * 8 + i], bf2f(e[i])));
    }
    return a;
}

// LIN: 0 q|k|v, 1 o, 2 gate|up, 3 down.  Grid (tiles, slices), cluster (1, slices).
// Dynamic shared memory: W atoms | adapter atoms (AD) | x atoms; then the partial sums in their place.
template <int LIN, bool AD, int DH>
__global__ void __launch_bounds__(ST_THREADS, 1)
    k_step_linear(const __grid_constant__ StepArgs a, const __grid_constant__ StepLin w) {
    constexpr bool NORM = LIN == 0 || LIN == 2;  // the operand is RMSNorm(h)
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
            for (int q = ct; q < TILE_ROWS * cpr; q += ST_STAGERS) {
                const int j = q / cpr, e = q % cpr;
                const int f = LIN == 2 ? (j < 64 ? tile * 64 + j : dm.I + tile * 64 + (j - 64)) : ft + j;
                S.brows[j * cpr + (j >> 2) + e] = __ldg(reinterpret_cast<const uint4 *>(w.lora_b + (size_t)f * r) + e);
            }
        }
        pdl_wait();
        if (NORM) {
            // ---- operand staging: the rows' chunks straight into the swizzled layout, then normalised in place
            // (as build_b in pass_kernel.cu)
            uint8_t *col = sX + (size_t)(c >> 3) * x_atom;
            auto chunk = [&](int at, int m) { return col + at * x_atom + m * 128 + (((c & 7) ^ (m & 7)) << 4); };
            bool ok = true;
            for (int hf = 0; hf < halves; ++hf) {
                const int at = (hf * ST_HALF) % ra;
                if (hf == 1 && ra == ST_HALF && !mbar_wait(&S.hdone, 0, a.status, DEV_TIMEOUT_MMA, &S.abort)) ok = false;
                if (!ok) break;
                const bf16 *src = a.h + (size_t)(slice * w.katoms + hf * ST_HALF) * KT + c * 8;
#pragma unroll 1
                for (int m = ct >> 5; m < M; m += ST_STAGERS / 32) cp_async16(chunk(at, m), src + (size_t)m * dm.H);
                cp_async_commit();
                if (hf == 0) {
                    const int nt = dm.H / TILE_ROWS;
                    for (int m = ct; m < M; m += ST_STAGERS) {
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
                        S.rs[m] = __fdiv_rn(1.0f, __fsqrt_rn(__fadd_rn(__fdiv_rn(sum, (float)dm.H), dm.eps)));
                    }
                }
                cp_async_wait_all();
                if (hf == 0) bar_stagers();
                const __nv_bfloat162 *g2 = reinterpret_cast<const __nv_bfloat162 *>(&gv[hf]);
#pragma unroll 1
                for (int m = ct >> 5; m < M; m += ST_STAGERS / 32) {
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
                bar_stagers();
                if (ct == 0) mbarrier_arrive_one(&S.xfull[hf]);
            }
        }
    }
    __syncwarp();

    // ---- partial sums into shared memory (every MMA has read its operands): warps 4-7, one TMEM lane quarter
    // (32 features) each
    float *part = reinterpret_cast<float *>(base), *part_u = part + M * TILE_ROWS;
    if (warp >= 4) {
        const bool have = mbar_wait(&S.done, 0, a.status, DEV_TIMEOUT_MMA, &S.abort) && !*(volatile int *)&S.abort;
        tc_fence_after();
        const int q = warp - 4, row = q * 32 + lane;
        const uint32_t tq = tmem + ((uint32_t)(q * 32) << 16);
        for (int c0 = 0; have && c0 < M; c0 += 16) {
            uint32_t v[16];
            tmem_ld_16cols(tq + (uint32_t)c0, v);
            tmem_ld_wait();
#pragma unroll
            for (int j = 0; j < 16; ++j)
                if (c0 + j < M) part[(c0 + j) * TILE_ROWS + row] = __uint_as_float(v[j]);
            if (AD && q == 0) {
                tmem_ld_16cols(tq + (uint32_t)(a.bn + c0), v);
                tmem_ld_wait();
#pragma unroll
                for (int j = 0; j < 16; ++j)
                    if (c0 + j < M && lane < ru) part_u[(c0 + j) * ru + lane] = __uint_as_float(v[j]);
            }
        }
        tc_fence_before();
    }
    cluster_sync();
    if (warp == 0) tmem_dealloc(tmem, w.tmem_cols);
    if (warp < 2) pdl_wait();  // (the warps that have not yet; the stores below)

    // ---- rows slice, slice + slices, ...: one warp per row
    const uint32_t pa = smem_u32(part), pu = smem_u32(part_u) + 4u * (lane < ru ? lane : 0);
    float gn[4] = {0.f, 0.f, 0.f, 0.f};  // QK-norm gain of the lane's four features
    constexpr int LPH = DH / 4;          // lanes per head
    const int e0 = 4 * (lane % LPH);
    if (LIN == 0 && kind < 2) {
        const uint2 raw = __ldg(reinterpret_cast<const uint2 *>((kind == 0 ? w.q_norm : w.k_norm) + e0));
        const float2 x = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&raw.x));
        const float2 y = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&raw.y));
        gn[0] = x.x, gn[1] = x.y, gn[2] = y.x, gn[3] = y.y;
    }
    for (int m = slice + warp * w.ks; m < M; m += w.ks * (ST_THREADS / 32)) {
        float u[ST_RANK], u2[ST_RANK];  // the row's adapter intermediates (gate|up: gate's and up's)
        if (AD) {
            const float lu = rbf(sum_slices(pu + (uint32_t)(m * ru) * 4u, w.ks));  // lane j: u_j
            spread_u(lu, 0, u);
            if (LIN == 2) spread_u(lu, r, u2);
        }
        if constexpr (LIN == 2) {
            // gate rows 2l, 2l + 1 and up rows 64 + 2l, 64 + 2l + 1 -> act features 64 tile + 2l, + 2l + 1
            float g[2], up[2];
            {
                float2 gs = make_float2(0.f, 0.f), us = gs;
                const uint32_t ga = pa + (uint32_t)(m * TILE_ROWS + 2 * lane) * 4u;
                for (int s = 0; s < w.ks; ++s) {
                    const float2 x = ld_cluster_v2(map_cta(ga, s)), y = ld_cluster_v2(map_cta(ga + 256u, s));
                    gs = s == 0 ? x : make_float2(__fadd_rn(gs.x, x.x), __fadd_rn(gs.y, x.y));
                    us = s == 0 ? y : make_float2(__fadd_rn(us.x, y.x), __fadd_rn(us.y, y.y));
                }
                g[0] = gs.x, g[1] = gs.y, up[0] = us.x, up[1] = us.y;
            }
            float o[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                if (AD) {
                    g[e] = __fadd_rn(g[e], __fmul_rn(dm.lora_scale, lora_dot_s(u, S.brows, 2 * lane + e, r)));
                    up[e] = __fadd_rn(up[e], __fmul_rn(dm.lora_scale, lora_dot_s(u2, S.brows, 64 + 2 * lane + e, r)));
                }
                const float gt = rbf(g[e]);
                o[e] = __fmul_rn(__fdiv_rn(gt, __fadd_rn(1.0f, expf(-gt))), rbf(up[e]));
            }
            *reinterpret_cast<uint32_t *>(a.act + (size_t)m * dm.I + tile * 64 + 2 * lane) = pack_bf162(o[0], o[1]);
        } else {
            uint2 hraw = make_uint2(0, 0);
            uint2 *hp = reinterpret_cast<uint2 *>(a.h + (size_t)m * dm.H + ft) + lane;
            if (LIN == 1 || LIN == 3) hraw = __ldcg(hp);
            const float4 y4 = sum_slices4(pa + (uint32_t)(m * TILE_ROWS + 4 * lane) * 4u, w.ks);
            float y[4] = {y4.x, y4.y, y4.z, y4.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if (AD) y[e] = __fadd_rn(y[e], __fmul_rn(dm.lora_scale, lora_dot_s(u, S.brows, 4 * lane + e, r)));
                y[e] = rbf(y[e]);
            }
            if constexpr (LIN == 0) {
                const int b = a.pd.b0 + m / a.pd.R, pos = a.L[b] + m % a.pd.R, pg = pos / PAGE;
                const int head = (ft - (kind == 0 ? 0 : (kind == 1 ? qw : qw + kvw))) / DH + lane / LPH;
                bool bad = kind > 0 && pg >= a.kv.pages_per_seq;
                if (kind < 2) {
                    bad = bad || pos >= a.rope_rows;
                    float ssq = __fmul_rn(y[0], y[0]);
#pragma unroll
                    for (int j = 1; j < 4; ++j) ssq = __fadd_rn(ssq, __fmul_rn(y[j], y[j]));
#pragma unroll
                    for (int off = LPH / 2; off >= 1; off >>= 1) ssq = __fadd_rn(ssq, __shfl_xor_sync(0xffffffffu, ssq, off));
                    const float rs = __fdiv_rn(1.0f, __fsqrt_rn(__fadd_rn(__fdiv_rn(ssq, (float)DH), dm.eps)));
                    const float4 *c4 = reinterpret_cast<const float4 *>(a.rope_cs + (size_t)(bad ? 0 : pos) * (DH / 2) + (e0 % (DH / 2)));
                    const float4 ca = __ldg(c4), cb = __ldg(c4 + 1);
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
                if (kind > 0) {
                    const int page = a.kv.page_table[b * a.kv.pages_per_seq + pg];
                    dst = static_cast<bf16 *>(kind == 1 ? a.kv.k : a.kv.v) +
                          ((((size_t)w.layer * a.kv.n_pages + page) * dm.Hkv + head) * PAGE + (pos % PAGE)) * DH + e0;
                }
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
    cluster_sync();  // no CTA leaves while another still reads its partials
}

// ------------------------------------------------------------------ attention step
//
// Grid (CTAs per group, KV heads, sequences).  CTA `rank` of a (sequence, KV head) takes splits rank,
// rank + cs, ... of 128 keys, up to two staged at a time; units of one 16-row query tile against one split
// (or 64-key half of it) go to the warps, as in attn_split (pass_kernel.cu).
//
// CLUSTER: the group's CTAs are a cluster.  The partial results (m, l, O) stay in shared memory, and
// after the cluster barrier the CTAs merge rows rank, rank + cs, ... in key order.  Otherwise (more
// splits than a portable cluster has CTAs, or more groups than the GPU holds clusters of: then clusters
// wait for one another's SMs) every split is a CTA of its own, the partial results go to memory and
// k_step_merge merges them.
constexpr int SA_WARPS = 8;   // compute warps of a cluster's CTA (two splits' units)
constexpr int SG_WARPS = 4;   // compute warps of a single split's CTA
constexpr int SA_STATS = 4;   // partial results per row at most: 32 x this

template <int DH>
struct SaLayout {
    static constexpr int SPB = 2 * (DH / 64) * ATT_SUB_BYTES;  // K, then V of a split
    static constexpr int PITCH = DH + 4;                       // floats per partial row
};

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
__global__ void __launch_bounds__(32 * (CLUSTER ? SA_WARPS : SG_WARPS) + 32, CLUSTER ? 1 : 2)
    k_step_attn(const __grid_constant__ CUtensorMap kmap, const __grid_constant__ CUtensorMap vmap,
                const __grid_constant__ StepArgs a, int layer, int bufs, int parts) {
    using LY = SaLayout<DH>;
    constexpr int WARPS = CLUSTER ? SA_WARPS : SG_WARPS;
    constexpr int KS = DH / 16, DT = DH / 8, SUBS = DH / 64, NP = ATT_SPLIT / PAGE;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ uint64_t full[2], empty[2];
    __shared__ int s_abort;
    const Dims &dm = a.dm;
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int rank = blockIdx.x, cs = gridDim.x, g = blockIdx.y, bl = blockIdx.z;
    const int b = a.pd.b0 + bl, R = a.pd.R, grp = dm.Hq / dm.Hkv, RH = R * grp;
    const int sub_sh = a.att_subs - 1, HALF = ATT_SPLIT >> sub_sh;          // one or two partial results per split
    float *po = reinterpret_cast<float *>(base + bufs * LY::SPB);           // [parts][RH][PITCH]
    float2 *pml = reinterpret_cast<float2 *>(po + (size_t)parts * RH * LY::PITCH);  // [parts][RH]
    if (threadIdx.x == 0) {
        for (int i = 0; i < 2; ++i) {
            mbar_init(&full[i], 1);
            mbar_init(&empty[i], WARPS);
        }
        s_abort = 0;
        fence_mbarrier_init();
        prefetch_tensormap(&kmap);
        prefetch_tensormap(&vmap);
    }
    __syncthreads();
    pdl_launch();
    // the cached length was set by a kernel that finished before this pass began
    const int L = a.L[b], T = L + R, nsp = (T + ATT_SPLIT - 1) / ATT_SPLIT;
    const int mine = rank < nsp ? (nsp - 1 - rank) / cs + 1 : 0;  // splits of this CTA

    if (warp == WARPS) {
        // ---- producer warp: lane p the page p of a split.  Pages entirely below L hold earlier passes' keys
        // and are requested at once; the block's own after the wait (their page ids are read before it).
        auto page_of = [&](int j) {
            const int s = rank + j * cs, p = s * NP + lane;
            return lane < NP && p * PAGE < T && p < a.kv.pages_per_seq ? a.kv.page_table[(size_t)b * a.kv.pages_per_seq + p] : -1;
        };
        auto request = [&](int j, int buf, int page, bool cached) {
            const int kp = (rank + j * cs) * ATT_SPLIT + lane * PAGE;
            const unsigned mask = __ballot_sync(0xffffffffu, page >= 0 && (kp + PAGE <= L) == cached);
            const uint32_t bytes = (uint32_t)__popc(mask) * 2u * SUBS * PAGE * 128u;
            if (lane == 0) {
                if (!cached)
                    mbar_arrive_expect_tx(&full[buf], bytes);
                else if (bytes)
                    mbar_expect_tx(&full[buf], bytes);
            }
            __syncwarp();
#pragma unroll 1
            for (int c0 = 0; c0 < NP * 2 * SUBS; c0 += 32) {
                const int cp = c0 + lane, p = cp / (2 * SUBS), q = cp % (2 * SUBS);
                const int pg = __shfl_sync(0xffffffffu, page, p & 31);
                if (p < NP && ((mask >> p) & 1u))
                    tma_load_2d(base + buf * LY::SPB + q * ATT_SUB_BYTES + p * PAGE * 128, q / SUBS ? &vmap : &kmap,
                                (q % SUBS) * 64, ((layer * a.kv.n_pages + pg) * dm.Hkv + g) * PAGE, &full[buf]);
            }
        };
        const int p0 = mine > 0 ? page_of(0) : -1, p1 = mine > 1 && bufs > 1 ? page_of(1) : -1;
        if (mine > 0) request(0, 0, p0, true);
        if (mine > 1 && bufs > 1) request(1, 1, p1, true);
        pdl_wait();
        fence_proxy_async_global();
        int j = 0;
        for (; j < mine; ++j) {
            const int buf = bufs > 1 ? j & 1 : 0;
            int page = j == 0 ? p0 : p1;
            if (j >= bufs) {
                page = page_of(j);
                if (!mbar_wait(&empty[buf], ((bufs > 1 ? j >> 1 : j) - 1) & 1, a.status, DEV_TIMEOUT_SLOT, &s_abort)) break;
                request(j, buf, page, true);
            }
            request(j, buf, page, false);
        }
        if (*(volatile int *)&s_abort)  // error path: the copies in flight get a bounded chance to land
            for (int h = j > bufs ? j - bufs : 0; h < j; ++h)
                mbar_wait(&full[bufs > 1 ? h & 1 : 0], (bufs > 1 ? h >> 1 : h) & 1, nullptr, 0, nullptr);
    } else {
        pdl_wait();
        const int gq = lane >> 2, tq = lane & 3, n_mt = (RH + 15) / 16;
        const float scale = a.att_scale;
        const uint32_t koff = attn_k_lane(lane), voff = attn_v_lane(lane);
        uint32_t ph = 0;
        for (int j0 = 0; j0 < mine; j0 += bufs, ph ^= 1) {
            const int nsx = min(bufs, mine - j0);
            bool landed = true;
            for (int i = 0; i < nsx; ++i)
                landed = landed && mbar_wait(&full[i], ph, a.status, DEV_TIMEOUT_LOAD, &s_abort);
            if (!landed) break;
#pragma unroll 1
            for (int unit = warp; unit < ((n_mt * nsx) << sub_sh); unit += WARPS) {
                // (nsx is 1 or 2)
                const int half = unit & sub_sh, us = unit >> sub_sh, sp = us & (nsx - 1), mt = us >> (nsx - 1), kb = half * HALF;
                const int k0 = (rank + (j0 + sp) * cs) * ATT_SPLIT;
                const uint32_t ka = smem_u32(base + sp * LY::SPB) + koff + kb * 128;
                const uint32_t va = smem_u32(base + sp * LY::SPB + SUBS * ATT_SUB_BYTES) + voff + kb * 128;
                const int qv0 = mt * 16 + gq, qv1 = qv0 + 8;
                const bool val0 = qv0 < RH, val1 = qv1 < RH;
                const int i0 = val0 ? qv0 / grp : 0, i1 = val1 ? qv1 / grp : 0;
                uint32_t qa[KS][4];
                {
                    const bf16 *q0 = a.q + ((size_t)(bl * R + i0) * dm.Hq + g * grp + (val0 ? qv0 % grp : 0)) * DH + 2 * tq;
                    const bf16 *q1 = a.q + ((size_t)(bl * R + i1) * dm.Hq + g * grp + (val1 ? qv1 % grp : 0)) * DH + 2 * tq;
#pragma unroll
                    for (int ks = 0; ks < KS; ++ks) {
                        qa[ks][0] = val0 ? __ldcg(reinterpret_cast<const unsigned *>(q0 + ks * 16)) : 0u;
                        qa[ks][1] = val1 ? __ldcg(reinterpret_cast<const unsigned *>(q1 + ks * 16)) : 0u;
                        qa[ks][2] = val0 ? __ldcg(reinterpret_cast<const unsigned *>(q0 + ks * 16 + 8)) : 0u;
                        qa[ks][3] = val1 ? __ldcg(reinterpret_cast<const unsigned *>(q1 + ks * 16 + 8)) : 0u;
                    }
                }
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
                    attn_scores<DH>(ka + c0 * 128, qa, sc);
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
                        attn_pv<DH>(va + (c0 + kstep * 16) * 128, pa, ma, mb, oc);
                    }
                }
                l0 += __shfl_xor_sync(0xffffffffu, l0, 1);
                l0 += __shfl_xor_sync(0xffffffffu, l0, 2);
                l1 += __shfl_xor_sync(0xffffffffu, l1, 1);
                l1 += __shfl_xor_sync(0xffffffffu, l1, 2);
                auto store = [&](bool val, int qv, int i, float m, float l, int e) {
                    if (!val) return;
                    float *dst;
                    if constexpr (CLUSTER) {
                        const int row = (((j0 + sp) << sub_sh) + half) * RH + qv;
                        dst = po + (size_t)row * LY::PITCH + 2 * tq;
                        if (tq == 0) pml[row] = make_float2(m, l);
                    } else {
                        const size_t row = ((size_t)(bl * R + i) * dm.Hq + g * grp + qv % grp) * a.att_splits_alloc +
                                           (((size_t)rank << sub_sh) + half);
                        dst = a.o_part + row * DH + 2 * tq;
                        if (tq == 0) a.ml_part[row] = make_float2(m, l);
                    }
#pragma unroll
                    for (int dt = 0; dt < DT; ++dt)
                        *reinterpret_cast<float2 *>(dst + dt * 8) = make_float2(oc[dt][e], oc[dt][e + 1]);
                };
                store(val0, qv0, i0, m0, l0, 0);
                store(val1, qv1, i1, m1, l1, 2);
            }
            __syncwarp();
            if (lane == 0)
                for (int i = 0; i < nsx; ++i) mbarrier_arrive_one(&empty[i]);
        }
    }
    if constexpr (CLUSTER) {
        __syncwarp();
        cluster_sync();
        if (warp < SA_WARPS) {
            const int cs_sh = __ffs(cs) - 1;  // (a power of two)
            const uint32_t poa = smem_u32(po), pma = smem_u32(pml);
            for (int qv = rank + warp * cs; qv < RH; qv += cs * SA_WARPS) {
                // partial p: split p >> sub_sh, the (split / cs)-th of CTA split % cs
                auto at = [&](uint32_t first, int p, uint32_t bytes) {
                    const int sp = p >> sub_sh;
                    return map_cta(first + (uint32_t)((((sp >> cs_sh) << sub_sh) + (p & sub_sh)) * RH + qv) * bytes, sp & (cs - 1));
                };
                merge_row<DH>(
                    nsp << sub_sh, lane, [&](int p) { return ld_cluster_v2(at(pma, p, 8u)); },
                    [&](int p, int c) { return ld_cluster_v4(at(poa, p, LY::PITCH * 4u) + (uint32_t)c * 4u); },
                    a.attn + ((size_t)(bl * R + qv / grp) * dm.Hq + g * grp + qv % grp) * DH);
            }
        }
        cluster_sync();  // no CTA leaves while another still reads its partials
    }
}

// One warp per (row, query head): merge of the partial results in memory.
template <int DH>
__global__ void __launch_bounds__(256) k_step_merge(const __grid_constant__ StepArgs a) {
    const int lane = threadIdx.x & 31, un = blockIdx.x * 8 + (threadIdx.x >> 5);
    const int m = un / a.dm.Hq;
    pdl_launch();
    const int T = m < a.pd.M ? a.L[a.pd.b0 + m / a.pd.R] + a.pd.R : 0;
    pdl_wait();
    if (m >= a.pd.M) return;
    const size_t row = (size_t)un * a.att_splits_alloc;
    merge_row<DH>(
        (T + ATT_SPLIT - 1) / ATT_SPLIT * a.att_subs, lane, [&](int p) { return __ldcg(a.ml_part + row + p); },
        [&](int p, int c) { return __ldcg(reinterpret_cast<const float4 *>(a.o_part + (row + p) * DH + c)); },
        a.attn + (size_t)un * DH);
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
    const float rs = __fdiv_rn(1.0f, __fsqrt_rn(__fadd_rn(__fdiv_rn(sum, (float)H), a.dm.eps)));
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

constexpr int ST_SMEM = 220 * 1024;   // dynamic shared memory of one CTA at most
constexpr int ST_MAX_CLUSTER = 16;

static int step_bn(int M) { return std::max(32, (M + 15) / 16 * 16); }

static int lin_smem(int bn, int ra, bool ad) { return ra * (TILE_BYTES + (ad ? ST_A_BYTES : 0) + bn * 128) + 1024; }

// ring atoms of a linear with katoms per slice (0: does not fit)
static int lin_ring(int bn, int M, int katoms, bool ad, int ru) {
    for (int ra : {katoms, ST_HALF}) {
        const int room = lin_smem(bn, ra, ad) - 1024;
        if (room + 1024 <= ST_SMEM && (int)sizeof(float) * M * (TILE_ROWS + ru) <= room) return ra;
    }
    return 0;
}

static int attn_smem(const Dims &dm, int R, int bufs, int parts) {
    const int rh = R * (dm.Hq / dm.Hkv);
    return bufs * 2 * (dm.d / 64) * ATT_SUB_BYTES + parts * rh * ((dm.d + 4) * 4 + 8) + 1024;
}

// The attention's form: cs CTAs of a cluster per (sequence, KV head) with bufs staged splits and `parts` partial
// results each, or cs = 0: one CTA per split and a merge kernel.  Clusters while each split gets its own
// CTA in a portable cluster, the partial results fit, and every cluster has its SMs at once.
static int attn_cluster(const Dims &dm, const PassDesc &pd, int subs, int nsplit, int *bufs, int *parts) {
    int c = 1;
    while (c < nsplit && c < 8) c *= 2;
    *bufs = std::min(2, (nsplit + c - 1) / c);
    *parts = (nsplit + c - 1) / c * subs;
    const bool ok = c >= nsplit && pd.nb * dm.Hkv * c <= gemm_ctas() && attn_smem(dm, pd.R, *bufs, *parts) <= ST_SMEM;
    return ok ? c : 0;
}

bool step_pass_fits(const Dims &dm, const PassDesc &pd, int subs, int nsplit) {
    const int K[4] = {dm.H, dm.Hq * dm.d, dm.H, dm.I};
    const int bn = step_bn(pd.M);
    if (pd.M > 256 || dm.r > ST_RANK) return false;
    for (int lin = 0; lin < 4; ++lin) {
        const int ka = mk_slice_atoms(lin, K[lin]);
        if (K[lin] / (ka * KT) > ST_MAX_CLUSTER) return false;
        if (lin_ring(bn, pd.M, ka, pd.adapter, pd.adapter ? (lin == 2 ? 2 : 1) * dm.r : 0) == 0) return false;
    }
    return nsplit * subs <= 32 * SA_STATS;  // (statistics a merging warp holds)
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

template <int DH>
static cudaError_t launch_lin(int lin, bool ad, dim3 grid, size_t smem, const StepArgs &a, const StepLin &w, cudaStream_t st) {
    const dim3 cl(1, grid.y);
#define STEP_LIN(L)                                                                                                      \
    return ad ? launch_step(k_step_linear<L, true, DH>, grid, cl, ST_THREADS, smem, st, a, w)                            \
              : launch_step(k_step_linear<L, false, DH>, grid, cl, ST_THREADS, smem, st, a, w)
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
    w.ring_atoms = lin_ring(a.bn, a.pd.M, w.katoms, ad, ad ? (lin == 2 ? 2 : 1) * a.dm.r : 0);
    if (w.ring_atoms == 0 || w.ks > ST_MAX_CLUSTER) return cudaErrorInvalidValue;
    w.tmem_cols = 32;
    while ((int)w.tmem_cols < (ad ? 2 : 1) * a.bn) w.tmem_cols <<= 1;
    if (lin == 1 || lin == 3)
        if (!encode_bf16_map(&w.xmap, lin == 1 ? (const void *)a.attn : (const void *)a.act, a.rows_alloc, w.K, a.bn))
            return cudaErrorInvalidValue;
    const dim3 grid(w.n_main / TILE_ROWS, w.ks);
    const size_t smem = lin_smem(a.bn, w.ring_atoms, ad);
    return a.dm.d == 128 ? launch_lin<128>(lin, ad, grid, smem, a, w, st) : launch_lin<64>(lin, ad, grid, smem, a, w, st);
}

template <int DH, bool BLK>
static cudaError_t launch_attn(const StepArgs &a, const CUtensorMap &kmap, const CUtensorMap &vmap, int layer, int nsplit,
                               cudaStream_t st) {
    int bufs, parts;
    const int cs = attn_cluster(a.dm, a.pd, a.att_subs, nsplit, &bufs, &parts);
    if (cs > 0)
        return launch_step(k_step_attn<DH, BLK, true>, dim3(cs, a.dm.Hkv, a.pd.nb), dim3(cs), 32 * SA_WARPS + 32,
                           attn_smem(a.dm, a.pd.R, bufs, parts), st, kmap, vmap, a, layer, bufs, parts);
    cudaError_t e = launch_step(k_step_attn<DH, BLK, false>, dim3(nsplit, a.dm.Hkv, a.pd.nb), dim3(1), 32 * SG_WARPS + 32,
                                attn_smem(a.dm, a.pd.R, 1, 0), st, kmap, vmap, a, layer, 1, 0);
    if (e != cudaSuccess) return e;
    return launch_pdl(k_step_merge<DH>, (a.pd.M * a.dm.Hq + 7) / 8, 256, 0, st, a);
}

cudaError_t launch_step_attn(const StepArgs &a, const CUtensorMap &kmap, const CUtensorMap &vmap, int layer, int nsplit,
                             cudaStream_t st) {
    const bool blk = a.pd.mask_mode == MASK_BLOCK_DRAFT;
    if (a.dm.d == 128)
        return blk ? launch_attn<128, true>(a, kmap, vmap, layer, nsplit, st) : launch_attn<128, false>(a, kmap, vmap, layer, nsplit, st);
    return blk ? launch_attn<64, true>(a, kmap, vmap, layer, nsplit, st) : launch_attn<64, false>(a, kmap, vmap, layer, nsplit, st);
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
    };
#define STEP_SET(L)                               \
    set((const void *)k_step_linear<L, true, 128>);  \
    set((const void *)k_step_linear<L, false, 128>); \
    set((const void *)k_step_linear<L, true, 64>);   \
    set((const void *)k_step_linear<L, false, 64>)
    STEP_SET(0);
    STEP_SET(1);
    STEP_SET(2);
    STEP_SET(3);
#undef STEP_SET
#define STEP_SET(DH, BLK)                            \
    set((const void *)k_step_attn<DH, BLK, true>);   \
    set((const void *)k_step_attn<DH, BLK, false>)
    STEP_SET(128, true);
    STEP_SET(128, false);
    STEP_SET(64, true);
    STEP_SET(64, false);
#undef STEP_SET
    return e;
}

}  // namespace pbd
