// linear_op.cu -- the standalone block linear of few rows, or of few columns and a long K (include/pbd_ops.h), in one
// kernel.
//
//     y = bf16(x W^T + scale * bf16(x A^T) B^T),   x [M, K], W [N, K], A [r, K], B [N, r]
//
// W and A are read where the caller has them: a 2-D tiled TMA load with the 128-byte swizzle turns
// a 128 x 64 box of a row-major matrix into the tensor core's operand tile, so no re-tiled copy of
// the weight is made (that copy cost a clear, a read and a write of the weight before the kernel
// read it a third time).
//
// Grid (N / 128 row tiles, slice CTAs, blocks of 64 token rows).  A tile's K slices (256 wide) go to the CTAs of one
// thread-block cluster: CTA c of cs takes slices c, c + cs, ..., one group of cs slices after the other.  For
// a slice it multiplies its weight box by the token rows into one accumulator and the adapter's A rows by
// the same rows into a second one, and leaves both as fp32 partial sums in its shared memory.  After a
// cluster barrier CTA c takes rows c, c + cs, ...: it reads the group's partials through distributed
// shared memory and adds them in slice order, so a row's bits depend neither on M nor on timing.
//
// Bound: latency.  GPU time at M = 17, r = 16 (cold caches): 8.8 us for K = 1024, N = 6144 and 8.5 us for
// K = 3072, N = 1024; 6.7 us at M = 1, K = 2048, N = 1024, r = 0.  With one CTA an SM, as before the adapter's place
// was cut to its rank, the first took 13.2.  With the partial sums in global memory and the last CTA of a tile
// finishing it alone: 22.0, 17.4 and 8.2 us, of which 8 us that last step; as re-tiling, split-K and
// reduction kernels: 21.4, 20.5 and 12.5 us and their gaps.
#include <algorithm>

#include "common.cuh"
#include "pbd_internal.h"

namespace pbd {

constexpr int LO_THREADS = 256;
constexpr int LO_MAX_STAGES = 4;
constexpr int LO_SMEM_HALF = 112 * 1024;  // dynamic shared memory with which two CTAs share an SM
constexpr int LO_SMEM_MAX = 224 * 1024;

// Dynamic shared memory: `stages` of W tile, 16 KiB | x tile, bn x 128 bytes | adapter rows, whole KiB; then the
// tile's B rows, transposed and widened, [r][128]; then, with several groups, the partial sums [rows][128]
// and [rows][r] (one group: they take the ring's place).  The adapter's MMA reads 128 rows from its r rows on:
// what follows them reaches only accumulator rows that nobody reads.
struct LoSmem {
    int a_bytes, stage, b_off, part_off, total;
    LoSmem(int bn, int r, int rows, int groups, int stages) {
        a_bytes = (r * 128 + 1023) / 1024 * 1024;
        stage = TILE_BYTES + bn * 128 + a_bytes;
        const int ring = stages * stage, part = (rows * (TILE_ROWS + r) * 4 + 15) / 16 * 16;
        b_off = groups > 1 || ring > part ? ring : part;
        part_off = groups > 1 ? b_off + r * TILE_ROWS * 4 : 0;
        total = b_off + r * TILE_ROWS * 4 + (groups > 1 ? part : 0);
        if (r > 0 && total < ring - a_bytes + TILE_BYTES) total = ring - a_bytes + TILE_BYTES;
    }
};

// ONE: one group.
template <bool ONE>
__global__ void __launch_bounds__(LO_THREADS, 2) k_linear_op(const __grid_constant__ LinOpArgs a) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ uint64_t full[LO_MAX_STAGES], empty[LO_MAX_STAGES], done, drain;
    __shared__ uint32_t tmem_slot;
    __shared__ int s_abort;
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int tile = blockIdx.x, rank = blockIdx.y, tok0 = blockIdx.z * LINEAR_OP_ROWS, rows = min(a.M - tok0, LINEAR_OP_ROWS);
    const int groups = ONE ? 1 : a.groups;
    const int stage = a.stage, x_off = TILE_BYTES, a_off = TILE_BYTES + a.bn * 128;
    const uint32_t s_b = smem_u32(base + a.b_off);
    const uint32_t tmem_cols = (uint32_t)(a.r > 0 ? 2 * a.bn : a.bn);  // one or two accumulators of 32 or 64 columns
    if (threadIdx.x == 0) {
        for (int s = 0; s < LO_MAX_STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(&done, 1);
        mbar_init(&drain, 1);
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
    const int mine = ONE ? 1 : (a.ks - 1 - rank) / a.cs + 1;  // this CTA's slices
    const int atoms = mine * a.kt_per;

    const uint32_t part = smem_u32(base + a.part_off), part_u = part + (uint32_t)(rows * TILE_ROWS) * 4u;
    const uint32_t pa = part + 16u * lane, ua = part_u + 4u * (lane < a.r ? lane : 0);

    // partial sums of row m over the group's n slices, in slice order, onto (y, u)
    auto fold = [&](int m, int n, bool first, float4 &y, float &u) {
        constexpr int QB = 4;  // slices whose loads are in flight together
        for (int q0 = 0; q0 < n; q0 += QB) {
            float4 v[QB];
            float w[QB];
#pragma unroll
            for (int q = 0; q < QB; ++q) {
                const int rk = min(q0 + q, n - 1);
                v[q] = ld_cluster_v4(map_cta(pa + (uint32_t)(m * TILE_ROWS) * 4u, rk));
                w[q] = a.r > 0 ? ld_cluster(map_cta(ua + (uint32_t)(m * a.r) * 4u, rk)) : 0.f;
            }
#pragma unroll
            for (int q = 0; q < QB; ++q) {
                if (q0 + q >= n) break;
                if (first && q0 + q == 0) {
                    y = v[0];
                    u = w[0];
                } else {
                    y = make_float4(__fadd_rn(y.x, v[q].x), __fadd_rn(y.y, v[q].y), __fadd_rn(y.z, v[q].z),
                                    __fadd_rn(y.w, v[q].w));
                    u = __fadd_rn(u, w[q]);
                }
            }
        }
    };
    // the adapter's delta and the stores: lane l features 4l..4l+3
    auto finish = [&](int m, float4 y, float u) {
        if (a.r > 0) {
            u = rbf(u);
            float4 d = make_float4(0.f, 0.f, 0.f, 0.f);
            for (int j = 0; j < a.r; ++j) {
                const float uj = __shfl_sync(0xffffffffu, u, j);
                const float4 b = ld_shared_v4(s_b + 16u * (uint32_t)(j * (TILE_ROWS / 4) + lane));
                d = make_float4(__fadd_rn(d.x, __fmul_rn(uj, b.x)), __fadd_rn(d.y, __fmul_rn(uj, b.y)),
                                __fadd_rn(d.z, __fmul_rn(uj, b.z)), __fadd_rn(d.w, __fmul_rn(uj, b.w)));
            }
            y = make_float4(__fadd_rn(y.x, __fmul_rn(a.scale, d.x)), __fadd_rn(y.y, __fmul_rn(a.scale, d.y)),
                            __fadd_rn(y.z, __fmul_rn(a.scale, d.z)), __fadd_rn(y.w, __fmul_rn(a.scale, d.w)));
        }
        const int f = tile * TILE_ROWS + 4 * lane;
        if (f >= a.N) return;
        bf16 *dst = a.y + (size_t)(tok0 + m) * a.N + f;
        if (a.vec_store) {
            *reinterpret_cast<uint2 *>(dst) = make_uint2(pack_bf162(y.x, y.y), pack_bf162(y.z, y.w));
        } else {
            dst[0] = f2bf(y.x);
            dst[1] = f2bf(y.y);
            dst[2] = f2bf(y.z);
            dst[3] = f2bf(y.w);
        }
    };

    // (producer: atoms requested so far, the next one's K and its place in the slice, ring slot and phase; a fresh
    // barrier counts as having completed the phase before its first.  MMA issuer: atoms consumed, slot, phase.)
    int sent = 0, slot = 0, k0 = rank * a.kt_per * KT, in = 0;
    bool dead = false;
    uint32_t ph = warp == 0 ? 1 : 0;
    float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
    float u = 0.f;
    for (int g = 0; g < groups; ++g) {
        if (warp == 0 && elect_one()) {
            // this group's atoms, and of the next group's what the ring takes once this one's are consumed (no more: the
            // next group's MMAs come after this group's barriers, which this thread has to reach)
            const uint32_t bytes = (uint32_t)TILE_BYTES + (uint32_t)a.r * 128u + (uint32_t)a.bn * 128u;
            const int end = ONE ? atoms : min(atoms, (g + 1) * a.kt_per + a.stages);
            for (; !dead && sent < end; ++sent) {
                if (!mbar_wait(&empty[slot], ph, a.status, DEV_TIMEOUT_SLOT, &s_abort)) break;
                uint8_t *st = base + slot * stage;
                mbar_arrive_expect_tx(&full[slot], bytes);
                tma_load_2d(st, &a.wmap, k0, tile * TILE_ROWS, &full[slot]);
                if (a.r > 0) tma_load_2d(st + a_off, &a.amap, k0, 0, &full[slot]);
                tma_load_2d(st + x_off, &a.xmap, k0, tok0, &full[slot]);
                if (++slot == a.stages) slot = 0, ph ^= 1;
                k0 += KT;
                if (!ONE && ++in == a.kt_per) in = 0, k0 += (a.cs - 1) * a.kt_per * KT;
            }
            if (!dead && *(volatile int *)&s_abort) {  // error path: the copies in flight get a bounded chance to land
                for (int h = sent > a.stages ? sent - a.stages : 0; h < sent; ++h)
                    if (!mbar_wait(&full[h % a.stages], (h / a.stages) & 1, nullptr, 0, nullptr)) break;  // (all had this second)
                dead = true;
            }
        } else if (warp == 1 && (ONE || (g < mine && !dead)) && elect_one()) {
            const uint32_t idesc = idesc_bf16_f32(128, a.bn);
            tc_fence_after();  // (the group before has left the accumulators)
            for (int s = 0; s < a.kt_per; ++s, ++sent) {
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
                if (sent + a.stages < atoms) mma_commit(&empty[slot]);
                if (++slot == a.stages) slot = 0, ph ^= 1;
            }
            mma_commit(&done);
            if (*(volatile int *)&s_abort) {  // error path: every MMA issued completes before TMEM goes
                mma_commit(&drain);
                mbar_wait(&drain, 0, nullptr, 0, nullptr);
                dead = true;
            }
        } else if (warp >= 2 && a.r > 0 && g == 0) {
            // the tile's B rows, transposed, while the operands stream in; a thread's loads go out together (one at a
            // time they took 3 us at rank 16)
            constexpr int LB = 12, T = LO_THREADS - 64;
            const bf16 *b = a.b + (size_t)tile * TILE_ROWS * a.r;
            const int n = TILE_ROWS * a.r;
            for (int i0 = threadIdx.x - 64; i0 < n; i0 += LB * T) {
                bf16 v[LB];
#pragma unroll
                for (int e = 0; e < LB; ++e) v[e] = __ldg(b + min(i0 + e * T, n - 1));
#pragma unroll
                for (int e = 0; e < LB; ++e) {
                    const int i = i0 + e * T;
                    if (i < n) st_shared(s_b + 4u * (uint32_t)((i % a.r) * TILE_ROWS + i / a.r), bf2f(v[e]));
                }
            }
        }
        __syncwarp();
        // ---- partial sums into shared memory (one group: every MMA has read its operands): warps 4-7 own TMEM lanes
        // 0-31, ... = features of the tile, warp 0 reads the adapter's rows (lanes 0..r-1)
        if ((ONE || g < mine) && (warp >= 4 || (warp == 0 && a.r > 0))) {
            const bool have = mbar_wait(&done, g & 1, a.status, DEV_TIMEOUT_MMA, &s_abort) && !*(volatile int *)&s_abort;
            tc_fence_after();
            for (int c0 = 0; have && c0 < rows; c0 += 32) {
                uint32_t v[32];
                tmem_ld_32cols(tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(c0 + (warp == 0 ? a.bn : 0)), v);
                tmem_ld_wait();
                if (warp == 0) {
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        if (c0 + j < rows && lane < a.r) st_shared(part_u + 4u * (uint32_t)((c0 + j) * a.r + lane), __uint_as_float(v[j]));
                } else {
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        if (c0 + j < rows) st_shared(part + 4u * (uint32_t)((c0 + j) * TILE_ROWS + (int)threadIdx.x - 128), __uint_as_float(v[j]));
                }
            }
            tc_fence_before();
        }
        __syncwarp();
        cluster_sync();
        const int n = min(a.cs, a.ks - g * a.cs);
        if (ONE) {
            if (warp == 0) tmem_dealloc(tmem, tmem_cols);
            for (int m = rank + warp * a.cs; m < rows; m += a.cs * (LO_THREADS / 32)) {
                fold(m, n, true, y, u);
                finish(m, y, u);
            }
        } else if (rank + warp * a.cs < rows) {  // (one row a warp: cs is at least 8)
            fold(rank + warp * a.cs, n, g == 0, y, u);
        }
        cluster_sync();  // no CTA overwrites its partials, or leaves, while another still reads them
    }
    if (!ONE) {
        if (warp == 0) tmem_dealloc(tmem, tmem_cols);
        if (rank + warp * a.cs < rows) finish(rank + warp * a.cs, y, u);
    }
}

cudaError_t configure_linear_op() {
    cudaError_t e = cudaSuccess;
    for (const void *f : {(const void *)k_linear_op<true>, (const void *)k_linear_op<false>}) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, LO_SMEM_MAX);
        if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    }
    return e;
}

int linear_op_bn(int M) { return M <= 32 ? 32 : 64; }

// CTAs of a tile's cluster: groups of as equal a size as it gets (17 slices: two of 9 and 8), but with several groups
// at least 8, so that each of 64 rows has a warp of its own.
static int lo_cluster(int ks) {
    static const int most = largest_cluster((const void *)k_linear_op<false>, LO_THREADS, LO_SMEM_MAX, LINEAR_OP_MAX_CLUSTER);
    const int groups = (ks + most - 1) / most;
    return groups == 1 ? ks : std::max(8, (ks + groups - 1) / groups);
}

// Per group: a chain of dependent steps, the slice's atoms, and the rows that a warp sums (and finishes) one after
// the other.  Measured: 5.1 us for one row and one atom, 7.0 for 64 rows, 10.4 for 64 with rank 16.
double linear_op_us(int M, int N, int ks, int kt_per, int r) {
    const int cs = lo_cluster(ks), groups = (ks + cs - 1) / cs, rows = std::min(M, LINEAR_OP_ROWS);
    const long ctas = (long)((N + TILE_ROWS - 1) / TILE_ROWS) * cs * ((M + LINEAR_OP_ROWS - 1) / LINEAR_OP_ROWS);
    const int turns = (rows + cs * (LO_THREADS / 32) - 1) / (cs * (LO_THREADS / 32));
    return (4.3 + 0.21 * kt_per + turns * (0.27 + 0.0225 * r)) * groups * std::max(1.0, (double)ctas / gemm_ctas());
}

cudaError_t launch_linear_op(LinOpArgs &a, cudaStream_t st) {
    a.bn = linear_op_bn(a.M);
    a.cs = lo_cluster(a.ks);
    a.groups = (a.ks + a.cs - 1) / a.cs;
    // Ring stages: as many as leave room for a second CTA on the SM (at least two), else all.  A CTA's time is that of its
    // dependent steps, so a second one beside it is worth more than stages (cold caches, 4096 x 4096, M = 64:
    // 24 us with two CTAs an SM, 37 with one; 17 rows, rank 16, 1024 x 6144: 8.8 and 13.2).
    const int rows = std::min(a.M, LINEAR_OP_ROWS), most = std::min(LO_MAX_STAGES, a.groups * a.kt_per);
    auto smem = [&](int stages) { return LoSmem(a.bn, a.r, rows, a.groups, stages).total + 1024; };
    for (a.stages = most; a.stages > std::min(most, 2) && smem(a.stages) > LO_SMEM_HALF;) --a.stages;
    if (smem(a.stages) > LO_SMEM_HALF) a.stages = most;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((a.N + TILE_ROWS - 1) / TILE_ROWS, a.cs, (a.M + LINEAR_OP_ROWS - 1) / LINEAR_OP_ROWS);
    cfg.blockDim = dim3(LO_THREADS);
    const LoSmem sm(a.bn, a.r, rows, a.groups, a.stages);
    a.stage = sm.stage;
    a.b_off = sm.b_off;
    a.part_off = sm.part_off;
    cfg.dynamicSmemBytes = sm.total + 1024;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1;
    attr[0].val.clusterDim.y = a.cs;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, a.groups == 1 ? k_linear_op<true> : k_linear_op<false>, a);
}

}  // namespace pbd
