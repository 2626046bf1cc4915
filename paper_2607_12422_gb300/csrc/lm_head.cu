// lm_head.cu -- the tied lm_head with greedy read-out, on the 5th-generation tensor core (sm_103a).
//
// A skinny contraction: M read-out rows (17 at batch 1, D = 16) against the [V, H] embedding, which
// is read exactly once per call.  The embedding supplies the 128-row MMA dimension and the tokens
// the N dimension:  D[vocabulary row, token] += E[row, k] * X[token, k]  (both K-major).  It is read
// either as pre-tiled 16 KiB tiles in the 128-byte swizzle layout (1-D bulk TMA; the decoder's copy)
// or straight from a row-major matrix (2-D tiled TMA, same swizzle).  A logit is one accumulation
// over all of H, so its bits do not depend on the number of rows.
//
// k_lm_head serves up to 64 rows with H <= 1024; beyond that the many-row kernel of gemm.cu does.
#include <algorithm>
#include <atomic>

#include "common.cuh"
#include "pbd_internal.h"

namespace pbd {

// One CTA per SM walks vocabulary tiles t = blockIdx.x, + gridDim.x, ...: the token rows'
// activation operand (all K atoms) is loaded once and stays in shared memory, weight tiles
// stream through a ring across tile boundaries, and two TMEM accumulators let the epilogue
// of one tile run under the MMAs of the next.  Warp 0 streams, warp 1 issues the MMAs, warps 2-5
// (one per TMEM lane quarter) store the logits and keep each token's best (value, lowest
// vocabulary row) over all tiles of the CTA: one redux.sync and one ballot per token and tile.
//
// Bound: HBM (311 MB for the 151936 x 1024 embedding).
constexpr int LMH_THREADS = 192;

template <int BN>
struct LmhLayout {
    static constexpr int STAGES = BN == 32 ? 8 : 5;  // with the token rows, what shared memory holds
    static constexpr int X_ATOM = BN * 128;  // one 64-wide K atom of the token rows
    static constexpr int RING_OFF = 0;
    static constexpr int X_OFF = STAGES * TILE_BYTES;
    static constexpr int MAX_ATOMS = 16;     // K <= 1024
    static constexpr int BAR_OFF = X_OFF + MAX_ATOMS * X_ATOM;
    static constexpr int RED_OFF = BAR_OFF + 256;
    static constexpr int RED_BYTES = 4 * BN * 8;  // [quarter][token] (value, index)
    static constexpr int TOTAL = RED_OFF + RED_BYTES + 1024;
    static constexpr uint32_t TMEM_COLS = 2 * BN < 32 ? 32 : 2 * BN;
};

template <int BN, bool TILED>
__global__ void __launch_bounds__(LMH_THREADS, 1)
    k_lm_head(const __grid_constant__ CUtensorMap xmap, const __grid_constant__ CUtensorMap wmap,
              const uint8_t *__restrict__ wtiles, int k_tiles, int n_tiles, int M, float *__restrict__ part_max,
              int *__restrict__ part_arg, float *__restrict__ logits, int V, int *status) {
    using LY = LmhLayout<BN>;
    constexpr int STAGES = LY::STAGES;
    extern __shared__ uint8_t smem_raw[];
    uint8_t *base = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    uint8_t *ring = base + LY::RING_OFF;
    uint8_t *sx = base + LY::X_OFF;
    uint64_t *full = reinterpret_cast<uint64_t *>(base + LY::BAR_OFF);
    uint64_t *empty = full + STAGES;
    uint64_t *x_full = empty + STAGES;
    uint64_t *acc_full = x_full + 1;   // [2]
    uint64_t *acc_empty = acc_full + 2;  // [2]
    uint64_t *drain = acc_empty + 2;
    uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(drain + 1);
    volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
    float *red_val = reinterpret_cast<float *>(base + LY::RED_OFF);
    int *red_idx = reinterpret_cast<int *>(red_val + 4 * BN);

    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    const int n_my = blockIdx.x < n_tiles ? (n_tiles - 1 - blockIdx.x) / gridDim.x + 1 : 0;

    if (threadIdx.x == 0) {
        for (int s = 0; s < STAGES; ++s) {
            mbar_init(&full[s], 1);
            mbar_init(&empty[s], 1);
        }
        mbar_init(x_full, 1);
        mbar_init(&acc_full[0], 1);
        mbar_init(&acc_full[1], 1);
        mbar_init(&acc_empty[0], 4);
        mbar_init(&acc_empty[1], 4);
        mbar_init(drain, 1);
        *abort_flag = 0;
        fence_mbarrier_init();
        prefetch_tensormap(&xmap);
        if (!TILED) prefetch_tensormap(&wmap);
    }
    if (warp == 0) tmem_alloc(tmem_slot, LY::TMEM_COLS);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *tmem_slot;

    if (warp == 0 && elect_one()) {
        // ---- producer: the token rows once, then the CTA's weight tiles back to back
        mbar_arrive_expect_tx(x_full, (uint32_t)(k_tiles * LY::X_ATOM));
        for (int a = 0; a < k_tiles; ++a) tma_load_2d(sx + a * LY::X_ATOM, &xmap, a * KT, 0, x_full);
        const uint64_t pol = l2_policy_evict_first();
        int g = 0, slot = 0;
        uint32_t ph = 1;  // (a fresh barrier counts as having completed the phase before its first)
        for (int j = 0; j < n_my && !*abort_flag; ++j) {
            const int tile = blockIdx.x + j * gridDim.x;
            for (int s = 0; s < k_tiles; ++s, ++g) {
                if (!mbar_wait(&empty[slot], ph, status, DEV_TIMEOUT_SLOT, abort_flag)) break;
                mbar_arrive_expect_tx(&full[slot], (uint32_t)TILE_BYTES);
                if (TILED)
                    bulk_g2s(ring + slot * TILE_BYTES, wtiles + ((size_t)tile * k_tiles + s) * TILE_BYTES, TILE_BYTES,
                             &full[slot], pol);
                else
                    tma_load_2d(ring + slot * TILE_BYTES, &wmap, s * KT, tile * TILE_ROWS, &full[slot]);
                if (++slot == STAGES) slot = 0, ph ^= 1;
            }
        }
        if (*abort_flag) {
            // error path: give the copies still in flight a bounded chance to land before exit
            mbar_wait(x_full, 0, nullptr, 0, nullptr);
            for (int h = g > STAGES ? g - STAGES : 0; h < g; ++h)
                mbar_wait(&full[h % STAGES], (h / STAGES) & 1, nullptr, 0, nullptr);
        }
    } else if (warp == 1 && elect_one()) {
        // ---- MMA issuer: per tile 4 x (128 x BN x 16) per K atom into accumulator j & 1
        const uint32_t idesc = idesc_bf16_f32(128, BN);
        bool ok = mbar_wait(x_full, 0, status, DEV_TIMEOUT_LOAD, abort_flag);
        tc_fence_after();
        int slot = 0;
        uint32_t ph = 0;
        for (int j = 0; ok && j < n_my; ++j) {
            const int acc = j & 1;
            if (j >= 2 && !mbar_wait(&acc_empty[acc], ((j >> 1) - 1) & 1, status, DEV_TIMEOUT_MMA, abort_flag)) break;
            tc_fence_after();
            const uint32_t d = tmem + (uint32_t)(acc * BN);
            for (int s = 0; s < k_tiles; ++s) {
                if (!mbar_wait(&full[slot], ph, status, DEV_TIMEOUT_LOAD, abort_flag)) {
                    ok = false;
                    break;
                }
                tc_fence_after();
                const uint64_t ad = sw128_kmajor_desc(ring + slot * TILE_BYTES);
                const uint64_t bd = sw128_kmajor_desc(sx + s * LY::X_ATOM);
#pragma unroll
                for (int kk = 0; kk < KT / 16; ++kk)
                    mma_bf16_ss(d, ad + 2ull * kk, bd + 2ull * kk, idesc, (s | kk) != 0 ? 1u : 0u);
                mma_commit(&empty[slot]);
                if (++slot == STAGES) slot = 0, ph ^= 1;
            }
            if (ok) mma_commit(&acc_full[acc]);
        }
        if (*abort_flag) {  // every MMA issued completes before TMEM is released
            mma_commit(drain);
            mbar_wait(drain, 0, nullptr, 0, nullptr);
        }
    } else if (warp >= 2) {
        // ---- epilogue: warp w reads TMEM lane quarter w % 4 (32 vocabulary rows)
        const int q = warp & 3;
        const int row = q * 32 + lane;
        float best[BN / 32];  // lane j: token c0 + j of each 32-token group
        int arg[BN / 32];
#pragma unroll
        for (int i = 0; i < BN / 32; ++i) best[i] = -INFINITY, arg[i] = 0x7fffffff;
        for (int j = 0; j < n_my; ++j) {
            const int acc = j & 1, tile = blockIdx.x + j * gridDim.x;
            if (!mbar_wait(&acc_full[acc], (j >> 1) & 1, status, DEV_TIMEOUT_MMA, abort_flag)) break;
            tc_fence_after();
            const int feat = tile * TILE_ROWS + row;
#pragma unroll
            for (int i = 0; i < BN / 32; ++i) {
                const int c0 = 32 * i;
                if (c0 >= M) break;
                uint32_t v[32];
                tmem_ld_32cols(tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * BN + c0), v);
                tmem_ld_wait();
                float bm = -INFINITY;
                int bl = -1;
#pragma unroll
                for (int jj = 0; jj < 32; ++jj) {
                    if (c0 + jj >= M) break;  // uniform across the warp
                    const float x = __uint_as_float(v[jj]);
                    if (logits != nullptr) logits[(size_t)(c0 + jj) * V + feat] = x;
                    int l;
                    const float m = warp_max(x, &l);
                    if (lane == jj) bm = m, bl = l;
                }
                // tiles come in ascending order: an equal later value never replaces
                const int idx = tile * TILE_ROWS + q * 32 + bl;
                if (bl >= 0 && (bm > best[i] || (bm == best[i] && idx < arg[i]))) best[i] = bm, arg[i] = idx;
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbarrier_arrive_one(&acc_empty[acc]);
        }
#pragma unroll
        for (int i = 0; i < BN / 32; ++i) {
            red_val[q * BN + 32 * i + lane] = best[i];
            red_idx[q * BN + 32 * i + lane] = arg[i];
        }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, LY::TMEM_COLS);
    for (int c = threadIdx.x; c < M; c += LMH_THREADS) {  // the four lane quarters
        float bv = red_val[c];
        int bi = red_idx[c];
#pragma unroll
        for (int w = 1; w < 4; ++w) {
            const float ov = red_val[w * BN + c];
            const int oi = red_idx[w * BN + c];
            if (ov > bv || (ov == bv && oi < bi)) bv = ov, bi = oi;
        }
        part_max[(size_t)blockIdx.x * M + c] = bv;
        part_arg[(size_t)blockIdx.x * M + c] = bi;
    }
}

// Every kernel's dynamic shared-memory limit, set once per device.
cudaError_t configure_linear_kernels() {
    static std::atomic<bool> done[64];
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 64 && done[dev].load()) return cudaSuccess;
    auto set = [&](const void *f, int bytes) {
        if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    };
    set((const void *)k_lm_head<32, true>, LmhLayout<32>::TOTAL);
    set((const void *)k_lm_head<32, false>, LmhLayout<32>::TOTAL);
    set((const void *)k_lm_head<64, true>, LmhLayout<64>::TOTAL);
    set((const void *)k_lm_head<64, false>, LmhLayout<64>::TOTAL);
    if (e == cudaSuccess) e = configure_linear_op();
    if (e == cudaSuccess) e = configure_gemm_kernels();
    if (e == cudaSuccess) e = configure_rows_kernels();
    if (e == cudaSuccess) e = configure_step_kernels();
    if (e == cudaSuccess && dev < 64) done[dev] = true;
    return e;
}

template <int BN>
static void launch_few(const CUtensorMap &x_map, const TiledWeight &w, const CUtensorMap *w_map, int grid, int M,
                       float *part_max, int *part_arg, float *logits, int *status, cudaStream_t st) {
    const int kt = w.K / KT, nt = w.n_main / TILE_ROWS;
    const uint8_t *tiles = static_cast<const uint8_t *>(w.tiles);
    if (tiles)
        k_lm_head<BN, true><<<grid, LMH_THREADS, LmhLayout<BN>::TOTAL, st>>>(x_map, x_map, tiles, kt, nt, M, part_max,
                                                                           part_arg, logits, w.n_main, status);
    else
        k_lm_head<BN, false><<<grid, LMH_THREADS, LmhLayout<BN>::TOTAL, st>>>(x_map, *w_map, tiles, kt, nt, M, part_max,
                                                                            part_arg, logits, w.n_main, status);
}

// a few rows over a short K: the kernel above (token rows resident in shared memory)
static bool few_rows(int M, int K) { return M <= 64 && K / KT <= LmhLayout<32>::MAX_ATOMS; }

int lm_head_box(int M, int K) { return few_rows(M, K) ? (M <= 32 ? 32 : 64) : (M + 15) / 16 * 16; }

cudaError_t launch_lm_head(const CUtensorMap &x_map, const TiledWeight &w, const CUtensorMap *w_map, int M,
                           float *tile_max, int *tile_arg, int *n_parts, float *logits, int *status, cudaStream_t st) {
    const int n_tiles = w.n_main / TILE_ROWS, grid = std::min(gemm_ctas(), n_tiles);
    if (grid <= 0 || M < 1 || M > 256) return cudaErrorInvalidValue;
    *n_parts = grid;
    if (few_rows(M, w.K)) {
        if (M <= 32)
            launch_few<32>(x_map, w, w_map, grid, M, tile_max, tile_arg, logits, status, st);
        else
            launch_few<64>(x_map, w, w_map, grid, M, tile_max, tile_arg, logits, status, st);
        return cudaGetLastError();
    }
    GemmArgs a{};
    a.xmap = x_map;
    if (w_map) a.wmap = *w_map;
    a.wt = static_cast<const uint8_t *>(w.tiles);
    a.k_tiles = a.slice_atoms = w.K / KT;
    a.n_slices = 1;
    a.f_tiles = n_tiles;
    a.bn = lm_head_box(M, w.K);
    a.M = M;
    a.rows = w.n_main;
    a.logits = logits;
    a.tile_max = tile_max;
    a.tile_arg = tile_arg;
    a.status = status;
    return launch_gemm(GEMM_HEAD, a, grid, st);
}

// Final argmax over the CTAs' partial results: lowest index among equal maxima.
__global__ void k_argmax_reduce(const float *__restrict__ tile_max, const int *__restrict__ tile_arg, int n_parts,
                                int rows, int *__restrict__ ids_out) {
    const int r = blockIdx.x;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    __shared__ float sv[8];
    __shared__ int si[8];
    float bv = -INFINITY;
    int bi = 0x7fffffff;
    for (int t = threadIdx.x; t < n_parts; t += blockDim.x) {
        const float v = tile_max[(size_t)t * rows + r];
        const int i = tile_arg[(size_t)t * rows + r];
        if (v > bv || (v == bv && i < bi)) {
            bv = v;
            bi = i;
        }
    }
    for (int off = 16; off >= 1; off >>= 1) {
        const float ov = __shfl_xor_sync(0xffffffffu, bv, off);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, off);
        if (ov > bv || (ov == bv && oi < bi)) {
            bv = ov;
            bi = oi;
        }
    }
    if (lane == 0) {
        sv[warp] = bv;
        si[warp] = bi;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        bv = sv[0];
        bi = si[0];
        for (int w = 1; w < (int)(blockDim.x >> 5); ++w)
            if (sv[w] > bv || (sv[w] == bv && si[w] < bi)) {
                bv = sv[w];
                bi = si[w];
            }
        ids_out[r] = bi;
    }
}

cudaError_t launch_argmax_reduce(const float *tile_max, const int *tile_arg, int n_parts, int rows, int *ids_out,
                                 cudaStream_t st) {
    if (rows <= 0) return cudaSuccess;
    k_argmax_reduce<<<rows, 256, 0, st>>>(tile_max, tile_arg, n_parts, rows, ids_out);
    return cudaGetLastError();
}

}  // namespace pbd
