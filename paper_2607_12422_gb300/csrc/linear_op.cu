// linear_op.cu -- the standalone block linear of few rows (include/pbd_ops.h), in one kernel.
//
//     y = bf16(x W^T + scale * bf16(x A^T) B^T),   x [M, K], W [N, K], A [r, K], B [N, r]
//
// W and A are read where the caller has them: a 2-D tiled TMA load with the 128-byte swizzle turns
// a 128 x 64 box of a row-major matrix into the tensor core's operand tile, so no re-tiled copy of
// the weight is made (that copy cost a clear, a read and a write of the weight before the kernel
// read it a third time).
//
// Grid (N / 128 row tiles, K slices of 256); the slices of a tile are one thread-block cluster.  A
// CTA multiplies its weight box by the token rows into one accumulator and the adapter's A rows
// by the same rows into a second one, and leaves both as fp32 partial sums in its shared memory.
// After the cluster barrier CTA s finishes rows s, s + slices, ...: it reads the slices' partials
// through distributed shared memory and adds them in slice order, so a row's bits depend neither on
// M nor on timing.
//
// Bound: latency.  GPU time at M = 17, r = 16 (cold caches): 13.5 us for K = 1024, N = 6144 and
// 9.1 us for K = 3072, N = 1024; 6.5 us at M = 1, K = 2048, N = 1024, r = 0.  With the partial sums in
// global memory and the last CTA of a tile finishing it alone: 22.0, 17.4 and 8.2 us, of which 8 us
// that last step; as re-tiling, split-K and reduction kernels: 21.4, 20.5 and 12.5 us and their gaps.
#include "common.cuh"
#include "pbd_internal.h"

namespace pbd {

constexpr int LO_THREADS = 256;
constexpr int LO_STAGES = 4;
constexpr int LO_MAX_R = 32;
constexpr int LO_A_BYTES = LO_MAX_R * 128;

// Dynamic shared memory: per stage the W tile, 16 KiB | x tile, bn x 128 bytes | with an adapter, its
// rows in 4 KiB.  The adapter's MMA reads 128 rows from there, 16 KiB: what follows the r rows (the next
// stage, or the 12 KiB kept behind the last one) reaches only accumulator rows that nobody reads.
// That keeps two CTAs on an SM.  The partial sums [M][128] and [M][r] take the ring's place afterwards.
__host__ __device__ inline int lo_stage_bytes(int bn, int r) { return TILE_BYTES + bn * 128 + (r > 0 ? LO_A_BYTES : 0); }

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
__device__ __forceinline__ float ld_cluster(uint32_t a) {
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
    return v;
}
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__global__ void __launch_bounds__(LO_THREADS, 2) k_linear_op(const __grid_constant__ LinOpArgs a) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ uint64_t full[LO_STAGES], empty[LO_STAGES], done;
    __shared__ uint32_t tmem_slot;
    __shared__ int s_abort;
    __shared__ float4 s_b[LO_MAX_R * TILE_ROWS / 4];  // B of the tile, [r][128], fp32
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int tile = blockIdx.x, slice = blockIdx.y;
    const int stage = lo_stage_bytes(a.bn, a.r), x_off = TILE_BYTES, a_off = TILE_BYTES + a.bn * 128;
    const uint32_t tmem_cols = a.bn <= 32 ? 64u : 128u;  // two accumulators of bn (32 or 64) columns
    if (threadIdx.x == 0) {
        for (int s = 0; s < LO_STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(&done, 1);
        s_abort = 0;
        fence_mbarrier_init();
        prefetch_tensormap(&a.xmap);
        prefetch_tensormap(&a.wmap);
    }
    if (warp == 0) tmem_alloc(&tmem_slot, tmem_cols);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_slot;

    if (warp == 0 && elect_one()) {
        const uint32_t bytes = (uint32_t)TILE_BYTES + (uint32_t)a.r * 128u + (uint32_t)a.bn * 128u;
        int s = 0, slot = 0, k0 = slice * a.kt_per * KT;
        uint32_t ph = 1;  // (a fresh barrier counts as having completed the phase before its first)
        for (; s < a.kt_per; ++s, k0 += KT) {
            if (!mbar_wait(&empty[slot], ph, a.status, DEV_TIMEOUT_SLOT, &s_abort)) break;
            uint8_t *st = base + slot * stage;
            mbar_arrive_expect_tx(&full[slot], bytes);
            tma_load_2d(st, &a.wmap, k0, tile * TILE_ROWS, &full[slot]);
            if (a.r > 0) tma_load_2d(st + a_off, &a.amap, k0, 0, &full[slot]);
            tma_load_2d(st + x_off, &a.xmap, k0, 0, &full[slot]);
            if (++slot == LO_STAGES) slot = 0, ph ^= 1;
        }
        if (*(volatile int *)&s_abort)  // error path: the copies in flight get a bounded chance to land
            for (int h = s > LO_STAGES ? s - LO_STAGES : 0; h < s; ++h)
                mbar_wait(&full[h % LO_STAGES], (h / LO_STAGES) & 1, nullptr, 0, nullptr);
    } else if (warp == 1 && elect_one()) {
        const uint32_t idesc = idesc_bf16_f32(128, a.bn);
        int slot = 0;
        uint32_t ph = 0;
        for (int s = 0; s < a.kt_per; ++s) {
            if (!mbar_wait(&full[slot], ph, a.status, DEV_TIMEOUT_LOAD, &s_abort)) break;
            tc_fence_after();
            const uint8_t *st = base + slot * stage;
            const uint64_t wd = sw128_kmajor_desc(st), xd = sw128_kmajor_desc(st + x_off);
#pragma unroll
            for (int kk = 0; kk < KT / 16; ++kk)
                mma_bf16_ss(tmem, wd + 2ull * kk, xd + 2ull * kk, idesc, (s | kk) != 0 ? 1u : 0u);
            if (a.r > 0) {
                const uint64_t ad = sw128_kmajor_desc(st + a_off);
#pragma unroll
                for (int kk = 0; kk < KT / 16; ++kk)
                    mma_bf16_ss(tmem + a.bn, ad + 2ull * kk, xd + 2ull * kk, idesc, (s | kk) != 0 ? 1u : 0u);
            }
            if (s + LO_STAGES < a.kt_per) mma_commit(&empty[slot]);
            if (++slot == LO_STAGES) slot = 0, ph ^= 1;
        }
        mma_commit(&done);  // also on the error path: every MMA issued completes before TMEM goes
    } else if (warp >= 2 && a.r > 0) {
        // the tile's B rows, transposed, while the operands stream in
        const bf16 *b = a.b + (size_t)tile * TILE_ROWS * a.r;
        float *sb = reinterpret_cast<float *>(s_b);
        for (int i = threadIdx.x - 64; i < TILE_ROWS * a.r; i += LO_THREADS - 64)
            sb[(i % a.r) * TILE_ROWS + i / a.r] = bf2f(b[i]);
    }
    __syncwarp();

    // ---- partial sums into shared memory (every MMA has read its operands): warp w < 4 owns TMEM
    // lanes 32w..32w+31 = features of the tile
    float *part = reinterpret_cast<float *>(base), *part_u = part + a.M * TILE_ROWS;
    const bool have = mbar_wait(&done, 0, a.status, DEV_TIMEOUT_MMA, &s_abort);
    tc_fence_after();
    if (warp < 4 && have && !*(volatile int *)&s_abort) {
        for (int c0 = 0; c0 < a.M; c0 += 32) {
            uint32_t v[32];
            tmem_ld_32cols(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, v);
            tmem_ld_wait();
#pragma unroll
            for (int j = 0; j < 32; ++j)
                if (c0 + j < a.M) part[(c0 + j) * TILE_ROWS + threadIdx.x] = __uint_as_float(v[j]);
            if (warp == 0 && a.r > 0) {  // adapter rows: lanes 0..r-1
                tmem_ld_32cols(tmem + (uint32_t)(a.bn + c0), v);
                tmem_ld_wait();
#pragma unroll
                for (int j = 0; j < 32; ++j)
                    if (c0 + j < a.M && lane < a.r) part_u[(c0 + j) * a.r + lane] = __uint_as_float(v[j]);
            }
        }
    }
    tc_fence_before();
    cluster_sync();
    if (warp == 0) tmem_dealloc(tmem, tmem_cols);
    // ---- rows slice, slice + slices, ...: one warp per row, lane l features 4l..4l+3
    const uint32_t pa = smem_u32(part) + 16u * lane, ua = smem_u32(part_u) + 4u * (lane < a.r ? lane : 0);
    for (int m = slice + warp * a.ks; m < a.M; m += a.ks * (LO_THREADS / 32)) {
        constexpr int QB = 4;  // slices whose loads are in flight together
        float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
        float u = 0.f;
        for (int q0 = 0; q0 < a.ks; q0 += QB) {
            float4 v[QB];
            float w[QB];
#pragma unroll
            for (int q = 0; q < QB; ++q) {
                const int rk = min(q0 + q, a.ks - 1);
                v[q] = ld_cluster_v4(map_cta(pa + (uint32_t)(m * TILE_ROWS) * 4u, rk));
                w[q] = a.r > 0 ? ld_cluster(map_cta(ua + (uint32_t)(m * a.r) * 4u, rk)) : 0.f;
            }
#pragma unroll
            for (int q = 0; q < QB; ++q) {
                if (q0 + q >= a.ks) break;
                if (q0 + q == 0) {
                    y = v[0];
                    u = w[0];
                } else {
                    y = make_float4(__fadd_rn(y.x, v[q].x), __fadd_rn(y.y, v[q].y), __fadd_rn(y.z, v[q].z),
                                    __fadd_rn(y.w, v[q].w));
                    u = __fadd_rn(u, w[q]);
                }
            }
        }
        if (a.r > 0) {
            u = rbf(u);
            float4 d = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int j = 0; j < a.r; ++j) {
                const float uj = __shfl_sync(0xffffffffu, u, j);
                const float4 b = s_b[j * (TILE_ROWS / 4) + lane];
                d = make_float4(__fadd_rn(d.x, __fmul_rn(uj, b.x)), __fadd_rn(d.y, __fmul_rn(uj, b.y)),
                                __fadd_rn(d.z, __fmul_rn(uj, b.z)), __fadd_rn(d.w, __fmul_rn(uj, b.w)));
            }
            y = make_float4(__fadd_rn(y.x, __fmul_rn(a.scale, d.x)), __fadd_rn(y.y, __fmul_rn(a.scale, d.y)),
                            __fadd_rn(y.z, __fmul_rn(a.scale, d.z)), __fadd_rn(y.w, __fmul_rn(a.scale, d.w)));
        }
        bf16 *dst = a.y + (size_t)m * a.N + tile * TILE_ROWS + 4 * lane;
        if (a.vec_store) {
            *reinterpret_cast<uint2 *>(dst) = make_uint2(pack_bf162(y.x, y.y), pack_bf162(y.z, y.w));
        } else {
            dst[0] = f2bf(y.x);
            dst[1] = f2bf(y.y);
            dst[2] = f2bf(y.z);
            dst[3] = f2bf(y.w);
        }
    }
    cluster_sync();  // no CTA leaves while another still reads its partials
}

cudaError_t configure_linear_op() {
    cudaError_t e = cudaFuncSetAttribute(k_linear_op, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         LO_STAGES * lo_stage_bytes(64, LO_MAX_R) + TILE_BYTES - LO_A_BYTES + 1024);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(k_linear_op, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    return e;
}

cudaError_t launch_linear_op(const LinOpArgs &a, cudaStream_t st) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(a.N / TILE_ROWS, a.ks);
    cfg.blockDim = dim3(LO_THREADS);
    cfg.dynamicSmemBytes = LO_STAGES * lo_stage_bytes(a.bn, a.r) + (a.r > 0 ? TILE_BYTES - LO_A_BYTES : 0) + 1024;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1;
    attr[0].val.clusterDim.y = a.ks;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, k_linear_op, a);
}

}  // namespace pbd
