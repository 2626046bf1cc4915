// gemm.cu -- tensor-core linears of many rows (more than one 64-row operand tile): the standalone
// linear and lm_head at large M, and the linears of prompt processing.
//
// As in every linear of this library the weight supplies the 128-row MMA dimension and the tokens
// the N dimension, and the sum over K is taken in slices (256 or 512 wide, fixed per linear): a
// slice accumulates in TMEM, and slices are added in fp32 in slice order.  An output element's
// bits therefore do not depend on M, on the token tile or on which of the kernels computed it:
// prompt rows equal the rows a decoding pass computes.
//
// Persistent CTAs walk 128-feature x bn-token tiles (bn chosen per call, up to 256).  Warp 0
// streams the operands of one 64-wide K atom per ring stage by TMA (weights either pre-tiled or
// straight from a row-major matrix), warp 1 issues the MMAs into two alternating TMEM accumulators, one
// slice each, and warps 4-11 keep the running sum of a tile in registers: they add slice s while
// the tensor core works on slice s + 1, and finish and store the tile while it works on the next
// tile's first two slices.  Split-K partial sums never touch memory.
#include <algorithm>

#include "common.cuh"
#include "pbd_internal.h"

namespace pbd {

constexpr int GM_EPI_WARPS = 8;
constexpr int GM_THREADS = 128 + 32 * GM_EPI_WARPS;  // three warpgroups
constexpr int GM_MAX_STAGES = 8;
constexpr int GM_MAX_BN = 256;
constexpr int GM_BUF = 256;  // TMEM columns per accumulator buffer
constexpr size_t GM_SMEM = 224 * 1024;

// two fp32 additions (round to nearest even, as __fadd_rn) in one instruction
__device__ __forceinline__ void add_f32x2(uint32_t &a0, uint32_t &a1, uint32_t b0, uint32_t b1) {
    asm("{\n\t.reg .b64 x, y;\n\tmov.b64 x, {%0, %1};\n\tmov.b64 y, {%2, %3};\n\tadd.rn.f32x2 x, x, y;\n\t"
        "mov.b64 {%0, %1}, x;\n\t}"
        : "+r"(a0), "+r"(a1)
        : "r"(b0), "r"(b1));
}

struct GemmState {
    uint64_t full[GM_MAX_STAGES], empty[GM_MAX_STAGES], acc_full[2], acc_empty[2], drain;
    uint32_t tmem_slot;
    int abort;
    // lm_head: best value and vocabulary row of each token per lane quarter
    float best[4][GM_MAX_BN];
    int arg[4][GM_MAX_BN];
    // per epilogue warp: a chunk of 16 tokens x 32 features on its way from feature-major registers
    // to 16-byte stores: words of two tokens, one row of 32 features per token pair, 16 bytes of padding
    uint4 turn[GM_EPI_WARPS][8 * 9];
};

template <int MODE, bool TILED>
__global__ void __launch_bounds__(GM_THREADS, 1) k_gemm(const __grid_constant__ GemmArgs a) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *ring = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    __shared__ GemmState S;
    const int warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), lane = threadIdx.x & 31;
    constexpr int A_BYTES = TILE_BYTES * (MODE == GEMM_GATE_UP ? 2 : 1);
    const int apg = a.stage_atoms, x_off = apg * A_BYTES, x_bytes = a.bn * 128;
    const int stage = x_off + apg * x_bytes, nst = a.stages;
    const int tiles = a.f_tiles * a.m_tiles;
    const int parts = a.n_slices + (a.delta ? 1 : 0);  // accumulation groups per tile
    if (threadIdx.x == 0) {
        for (int s = 0; s < nst; ++s) {
            mbar_init(&S.full[s], 1);
            mbar_init(&S.empty[s], 1);
        }
        for (int b = 0; b < 2; ++b) {
            mbar_init(&S.acc_full[b], 1);
            mbar_init(&S.acc_empty[b], GM_EPI_WARPS);
        }
        mbar_init(&S.drain, 1);
        S.abort = 0;
        fence_mbarrier_init();
        prefetch_tensormap(&a.xmap);
        if (!TILED) prefetch_tensormap(&a.wmap);
    }
    if (warp == 0) tmem_alloc(&S.tmem_slot, 2 * GM_BUF);
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = S.tmem_slot;

    pdl_launch();
    // Registers: the block starts with 3 x 128 threads x 168; the producer's warpgroup gives up
    // 128 x 128 of them and the two epilogue warpgroups take 128 x 56 each (40 + 2 x 224 <= 3 x 168),
    // which holds a tile's 128 running sums a thread without spills.
    if (warp < 4) {
        asm volatile("setmaxnreg.dec.sync.aligned.u32 40;");
        if (warp == 0 && elect_one()) {
            // ---- producer; weights that no second token tile reads need not stay in L2
            const uint64_t pol = a.m_tiles == 1 ? l2_policy_evict_first() : l2_policy_evict_normal();
            int slot = 0, issued = 0;
            uint32_t ph = 1;  // (a fresh barrier counts as having completed the phase before its first)
            bool ok = true;
            auto weights = [&](uint8_t *st, uint64_t *bar, int ft, int k) {
                if constexpr (MODE == GEMM_GATE_UP) {
                    // weight tile t holds gate rows 64t.. then up rows 64t..: two tiles make 128 of each
                    for (int e = 0; e < apg; ++e)
                        for (int j = 0; j < 2; ++j) {
                            const uint8_t *src = a.wt + ((size_t)(2 * ft + j) * a.k_tiles + k + e) * TILE_BYTES;
                            uint8_t *d = st + e * A_BYTES + j * (TILE_BYTES / 2);
                            bulk_g2s(d, src, TILE_BYTES / 2, bar, pol);
                            bulk_g2s(d + TILE_BYTES, src + TILE_BYTES / 2, TILE_BYTES / 2, bar, pol);
                        }
                } else if constexpr (TILED) {  // consecutive atoms of a weight tile are contiguous
                    bulk_g2s(st, a.wt + ((size_t)ft * a.k_tiles + k) * TILE_BYTES, (uint32_t)(apg * TILE_BYTES), bar, pol);
                } else {
                    for (int e = 0; e < apg; ++e)
                        tma_load_2d(st + e * A_BYTES, &a.wmap, (k + e) * KT, ft * TILE_ROWS, bar);
                }
            };
            // pre-tiled weights are a context's own and depend on nothing before this kernel: the first
            // stages' go out while that still runs (a caller's matrix may be what it writes)
            const int early = TILED ? min(nst, a.k_tiles / apg) : 0;
            for (int j = 0; j < early; ++j) {
                mbar_arrive_expect_tx(&S.full[j], (uint32_t)stage);
                weights(ring + j * stage, &S.full[j], blockIdx.x % a.f_tiles, j * apg);
            }
            pdl_wait();
            for (int t = blockIdx.x; ok && t < tiles; t += gridDim.x) {
                const int ft = t % a.f_tiles, tok0 = (t / a.f_tiles) * a.bn;
                for (int k = 0; k < a.k_tiles + (a.delta ? 1 : 0); k += apg) {
                    if (!mbar_wait(&S.empty[slot], ph, a.status, DEV_TIMEOUT_SLOT, &S.abort)) {
                        ok = false;
                        break;
                    }
                    uint8_t *st = ring + slot * stage;
                    uint64_t *bar = &S.full[slot];
                    if (++slot == nst) slot = 0, ph ^= 1;
                    ++issued;
                    if (k == a.k_tiles) {  // the adapter: B rows by u rows
                        mbar_arrive_expect_tx(bar, (uint32_t)(A_BYTES + x_bytes));
                        tma_load_2d(st, &a.bmap, 0, ft * TILE_ROWS, bar);
                        tma_load_2d(st + x_off, &a.umap, 0, tok0, bar);
                        continue;
                    }
                    if (issued > early) {
                        mbar_arrive_expect_tx(bar, (uint32_t)stage);
                        weights(st, bar, ft, k);
                    }
                    for (int e = 0; e < apg; ++e)
                        tma_load_2d(st + x_off + e * x_bytes, &a.xmap, (k + e) * KT, tok0, bar);
                }
            }
            if (*(volatile int *)&S.abort)  // error path: the copies in flight get a bounded chance to land
                for (int h = issued > nst ? issued - nst : 0; h < issued; ++h)
                    if (!mbar_wait(&S.full[h % nst], (h / nst) & 1, nullptr, 0, nullptr)) break;  // (all had this second)
        } else if (warp == 1 && elect_one()) {
            // ---- MMA issuer
            const uint32_t idesc = idesc_bf16_f32(128, a.bn);
            int slot = 0, p = 0;  // ring stage; accumulation groups so far
            uint32_t ph = 0;
            bool ok = true;
            for (int t = blockIdx.x; ok && t < tiles; t += gridDim.x) {
                for (int s = 0; ok && s < parts; ++s, ++p) {
                    const int buf = p & 1;
                    if (p >= 2 && !mbar_wait(&S.acc_empty[buf], ((p >> 1) - 1) & 1, a.status, DEV_TIMEOUT_MMA, &S.abort)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    const uint32_t d = tmem + (uint32_t)(buf * GM_BUF);
                    const bool dl = s == a.n_slices;
                    const int atoms = dl ? 1 : a.slice_atoms;
                    for (int k = 0; k < atoms; k += apg) {
                        if (!mbar_wait(&S.full[slot], ph, a.status, DEV_TIMEOUT_LOAD, &S.abort)) {
                            ok = false;
                            break;
                        }
                        tc_fence_after();
                        const uint8_t *st = ring + slot * stage;
                        uint64_t wd = sw128_kmajor_desc(st), xd = sw128_kmajor_desc(st + x_off);
                        if (dl) {  // K = 32: ranks up to 32, zero beyond the rank
#pragma unroll
                            for (int kk = 0; kk < 2; ++kk)
                                mma_bf16_ss(d, wd + 2ull * kk, xd + 2ull * kk, idesc, kk != 0 ? 1u : 0u);
                        } else {
#pragma unroll 1
                            for (int e = 0; e < apg; ++e, wd += A_BYTES / 16, xd += x_bytes / 16) {
#pragma unroll
                                for (int kk = 0; kk < KT / 16; ++kk)
                                    mma_bf16_ss(d, wd + 2ull * kk, xd + 2ull * kk, idesc, (k | e | kk) != 0 ? 1u : 0u);
                                if (MODE == GEMM_GATE_UP) {
                                    const uint64_t ud = wd + TILE_BYTES / 16;
#pragma unroll
                                    for (int kk = 0; kk < KT / 16; ++kk)
                                        mma_bf16_ss(d + a.bn, ud + 2ull * kk, xd + 2ull * kk, idesc, (k | e | kk) != 0 ? 1u : 0u);
                                }
                            }
                        }
                        mma_commit(&S.empty[slot]);
                        if (++slot == nst) slot = 0, ph ^= 1;
                    }
                    if (ok) mma_commit(&S.acc_full[buf]);
                }
            }
            if (*(volatile int *)&S.abort) {  // every MMA issued completes before TMEM is released
                mma_commit(&S.drain);
                mbar_wait(&S.drain, 0, nullptr, 0, nullptr);
            }
        }
    } else {
        asm volatile("setmaxnreg.inc.sync.aligned.u32 224;");
        pdl_wait();  // (the stores below)
        // ---- epilogue: warp w owns TMEM lane quarter w % 4 (32 features) and every other chunk of
        // 16 token columns
        const int q = warp & 3, hh = (warp - 4) >> 2;
        const uint32_t tq = tmem + ((uint32_t)(q * 32) << 16);
        const int row = q * 32 + lane;
        constexpr int NC = GM_MAX_BN / 32;                             // chunks per warp
        constexpr int GC = MODE == GEMM_GATE_UP ? NC / 2 : NC;         // of them gate (or plain) chunks
        float best[NC];
        int arg[NC];
        if (MODE == GEMM_HEAD)
#pragma unroll
            for (int i = 0; i < NC; ++i) best[i] = -INFINITY, arg[i] = 0x7fffffff;
        int p = 0;
        bool ok = true;
        for (int t = blockIdx.x; ok && t < tiles; t += gridDim.x) {
            const int ft = t % a.f_tiles, tok0 = (t / a.f_tiles) * a.bn;
            if constexpr (MODE == GEMM_HEAD) {
                const int buf = p & 1;
                if (!mbar_wait(&S.acc_full[buf], (p >> 1) & 1, a.status, DEV_TIMEOUT_MMA, &S.abort)) break;
                ++p;
                tc_fence_after();
                const int feat = ft * TILE_ROWS + row;
#pragma unroll
                for (int i = 0; i < NC; ++i) {
                    const int c = (2 * i + hh) * 16;
                    if (c >= a.M) break;  // uniform across the warp
                    uint32_t v[16];
                    tmem_ld_16cols(tq + (uint32_t)(buf * GM_BUF + c), v);
                    tmem_ld_wait();
                    float bm = -INFINITY;  // lane j < 16: the quarter's best of column c + j
                    int bl = -1;
#pragma unroll
                    for (int j = 0; j < 16; ++j) {
                        const float x = __uint_as_float(v[j]);
                        if (a.logits != nullptr && c + j < a.M) a.logits[(size_t)(c + j) * a.rows + feat] = x;
                        int l;
                        const float m = warp_max(x, &l);
                        if (lane == j) bm = m, bl = l;
                    }
                    // tiles come in ascending order: an equal later value never replaces
                    const int idx = ft * TILE_ROWS + q * 32 + bl;
                    if (bl >= 0 && (bm > best[i] || (bm == best[i] && idx < arg[i]))) best[i] = bm, arg[i] = idx;
                }
                tc_fence_before();
                __syncwarp();
                if (lane == 0) mbarrier_arrive_one(&S.acc_empty[buf]);
            } else {
                // No one thing bounds this kernel.  4096 x 1024 x 6144, us with the launch (8): 48.8; without the adds of
                // slices 47.7, with half the bytes of token rows 46.7, with neither 45.0; finished tiles not
                // rounded and stored 43.2.  Finishing a tile is the largest part: meanwhile the tensor core
                // has the next tile's first two slices and no more.  With a few instructions more per
                // element there it took twice as long, so the sums use the packed fp32 add and each kind of slice
                // has its own loop.
                uint32_t acc[NC][16];  // fp32 bits
                for (int s = 0; s < parts; ++s, ++p) {
                    const int buf = p & 1;
                    if (!mbar_wait(&S.acc_full[buf], (p >> 1) & 1, a.status, DEV_TIMEOUT_MMA, &S.abort)) {
                        ok = false;
                        break;
                    }
                    tc_fence_after();
                    // gate chunks then up chunks (GEMM_GATE_UP); chunk i of a kind: columns (2 i + hh) * 16
                    const uint32_t t0 = tq + (uint32_t)(buf * GM_BUF + hh * 16);
                    auto col = [&](int i) { return t0 + (uint32_t)(32 * (i % GC) + (i >= GC ? a.bn : 0)); };
                    auto on = [&](int i) { return 32 * (i % GC) + hh * 16 < a.bn; };  // (uniform)
                    if (s == 0) {
#pragma unroll
                        for (int i = 0; i < NC; ++i)
                            if (on(i)) tmem_ld_16cols(col(i), acc[i]);
                        tmem_ld_wait();
                    } else if (s < a.n_slices) {
#pragma unroll
                        for (int i = 0; i < NC; i += 2) {  // two chunks per round trip
                            uint32_t v[2][16];
#pragma unroll
                            for (int e = 0; e < 2; ++e)
                                if (on(i + e)) tmem_ld_16cols(col(i + e), v[e]);
                            tmem_ld_wait();
#pragma unroll
                            for (int e = 0; e < 2; ++e)
                                if (on(i + e))
#pragma unroll
                                    for (int j = 0; j < 16; j += 2) add_f32x2(acc[i + e][j], acc[i + e][j + 1], v[e][j], v[e][j + 1]);
                        }
                    } else {  // the adapter
#pragma unroll
                        for (int i = 0; i < NC; ++i) {
                            if (!on(i)) continue;
                            uint32_t v[16];
                            tmem_ld_16cols(col(i), v);
                            tmem_ld_wait();
#pragma unroll
                            for (int j = 0; j < 16; ++j)
                                acc[i][j] = __float_as_uint(__fadd_rn(__uint_as_float(acc[i][j]),
                                                                      __fmul_rn(a.scale, __uint_as_float(v[j]))));
                        }
                    }
                    tc_fence_before();
                    __syncwarp();
                    if (lane == 0) mbarrier_arrive_one(&S.acc_empty[buf]);
                }
                if (!ok) break;
                const int f = ft * TILE_ROWS + row;
                if (f - lane >= a.rows) continue;  // (uniform: rows is a multiple of 32)
                uint32_t *turn = reinterpret_cast<uint32_t *>(S.turn[warp - 4]);
                const int pr = lane >> 2, part = lane & 3;  // the lane's token pair and 8 features when storing
                bf16 *dst = a.y + (size_t)(tok0 + hh * 16 + 2 * pr) * a.ld + (f - lane) + 8 * part;
#pragma unroll
                for (int i = 0; i < GC; ++i) {
                    const int tok = tok0 + 32 * i + hh * 16;
                    if (32 * i + hh * 16 >= a.bn || tok >= a.M) break;
                    uint32_t w[8];  // tokens 2 j (low half) and 2 j + 1 of this lane's feature
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        float x[2];
#pragma unroll
                        for (int e = 0; e < 2; ++e) {
                            x[e] = __uint_as_float(acc[i][2 * j + e]);
                            if constexpr (MODE == GEMM_GATE_UP) {
                                const float gt = rbf(x[e]), up = rbf(__uint_as_float(acc[GC + i][2 * j + e]));
                                x[e] = __fmul_rn(__fdiv_rn(gt, __fadd_rn(1.0f, expf(-gt))), up);
                            }
                        }
                        w[j] = pack_bf162(x[0], x[1]);
                    }
                    if (!a.vec_store) {
#pragma unroll
                        for (int j = 0; j < 16; ++j)
                            if (tok + j < a.M)
                                a.y[(size_t)(tok + j) * a.ld + f] = __ushort_as_bfloat16((unsigned short)(w[j / 2] >> (16 * (j & 1))));
                        continue;
                    }
                    __syncwarp();  // the previous chunk has been read
#pragma unroll
                    for (int j = 0; j < 8; ++j) turn[j * 36 + lane] = w[j];
                    __syncwarp();
                    const uint4 u0 = *reinterpret_cast<const uint4 *>(turn + pr * 36 + 8 * part);
                    const uint4 u1 = *reinterpret_cast<const uint4 *>(turn + pr * 36 + 8 * part + 4);
                    bf16 *d = dst + (size_t)(32 * i) * a.ld;
                    if (tok + 2 * pr < a.M)
                        *reinterpret_cast<uint4 *>(d) = make_uint4(__byte_perm(u0.x, u0.y, 0x5410), __byte_perm(u0.z, u0.w, 0x5410),
                                                                   __byte_perm(u1.x, u1.y, 0x5410), __byte_perm(u1.z, u1.w, 0x5410));
                    if (tok + 2 * pr + 1 < a.M)
                        *reinterpret_cast<uint4 *>(d + a.ld) = make_uint4(__byte_perm(u0.x, u0.y, 0x7632), __byte_perm(u0.z, u0.w, 0x7632),
                                                                          __byte_perm(u1.x, u1.y, 0x7632), __byte_perm(u1.z, u1.w, 0x7632));
                }
            }
        }
        if (MODE == GEMM_HEAD && lane < 16)
#pragma unroll
            for (int i = 0; i < NC; ++i) {
                const int c = (2 * i + hh) * 16 + lane;
                if (c < GM_MAX_BN) S.best[q][c] = best[i], S.arg[q][c] = arg[i];
            }
    }
    tc_fence_before();
    __syncthreads();
    if (warp == 0) tmem_dealloc(tmem, 2 * GM_BUF);
    if (MODE == GEMM_HEAD)
        for (int c = threadIdx.x; c < a.M; c += GM_THREADS) {  // the four lane quarters
            float bv = S.best[0][c];
            int bi = S.arg[0][c];
#pragma unroll
            for (int w = 1; w < 4; ++w)
                if (S.best[w][c] > bv || (S.best[w][c] == bv && S.arg[w][c] < bi)) bv = S.best[w][c], bi = S.arg[w][c];
            a.tile_max[(size_t)blockIdx.x * a.M + c] = bv;
            a.tile_arg[(size_t)blockIdx.x * a.M + c] = bi;
        }
}

static int sm_count() {
    static int sms = 0;
    if (sms == 0) {
        int dev = 0, n = 0;
        if (cudaGetDevice(&dev) == cudaSuccess && cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess)
            sms = n;
    }
    return sms;
}

// Token tile width: the one that minimises waves x time of a tile on `ctas` CTAs.  A tile's time is its
// MMAs (cycles per 128 x bn x 16 instruction: 64 up to bn = 64, 67 at 128, 129 at 256, measured)
// plus about 3000 cycles to fill and drain the pipeline.
int gemm_pick_bn(int M, int f_tiles, int k_tiles, int max_bn, int ctas) {
    int best = 32;
    double best_t = 0;
    for (int bn = 32; bn <= max_bn; bn += 32) {
        const double mma = std::max(64.0, bn * 0.505);
        const long tiles = (long)f_tiles * ((M + bn - 1) / bn);
        const double t = (double)((tiles + ctas - 1) / ctas) * (k_tiles * 4.0 * mma + 3000.0);
        if (bn == 32 || t < best_t * 0.999) best = bn, best_t = t;
        if (bn >= M) break;
    }
    return best;
}

// Measured: 0.21 us an atom up to bn = 208 (K = 16384, one tile of 64 rows: 54 us), the MMAs' time above.
double gemm_us(int M, int f_tiles, int k_tiles, int bn) {
    const long tiles = (long)f_tiles * ((M + bn - 1) / bn), n = sm_count();
    return (double)((tiles + n - 1) / n) * (k_tiles * std::max(0.21, bn * 0.001) + 2.5);
}

template <int MODE, bool TILED>
static cudaError_t launch_one(GemmArgs &a, int ctas, cudaStream_t st) {
    // Atoms per ring stage: a stage costs the issuing threads about 200 ns of waiting, announcing and
    // committing whatever its size (measured), as long as the MMAs of one atom up to bn = 128; two
    // atoms share it where at least three stages still fit and slices hold whole stages.
    const int atom = TILE_BYTES * (MODE == GEMM_GATE_UP ? 2 : 1) + a.bn * 128;
    const int room = (int)(GM_SMEM - sizeof(GemmState) - 2048);
    a.stage_atoms = (a.slice_atoms % 2 == 0 && room / (2 * atom) >= 3) ? 2 : 1;
    const int stage = a.stage_atoms * atom;
    a.stages = std::min<int>(GM_MAX_STAGES, room / stage);
    const int grid = std::min(ctas, a.f_tiles * a.m_tiles);
    return launch_pdl(k_gemm<MODE, TILED>, grid, GM_THREADS, (size_t)a.stages * stage + 1024, st, a);
}

cudaError_t launch_gemm(GemmMode mode, GemmArgs &a, int ctas, cudaStream_t st) {
    const int n = ctas > 0 ? ctas : sm_count();
    if (n <= 0) return cudaErrorInvalidDevice;
    if (a.bn < 16 || a.bn > GM_MAX_BN || a.bn % 16 || (mode == GEMM_GATE_UP && a.bn > GM_MAX_BN / 2))
        return cudaErrorInvalidValue;
    a.m_tiles = (a.M + a.bn - 1) / a.bn;
    switch (mode) {
        case GEMM_Y: return a.wt ? launch_one<GEMM_Y, true>(a, n, st) : launch_one<GEMM_Y, false>(a, n, st);
        case GEMM_GATE_UP: return launch_one<GEMM_GATE_UP, true>(a, n, st);
        case GEMM_HEAD: return a.wt ? launch_one<GEMM_HEAD, true>(a, n, st) : launch_one<GEMM_HEAD, false>(a, n, st);
    }
    return cudaErrorInvalidValue;
}

int gemm_ctas() { return sm_count(); }

cudaError_t configure_gemm_kernels() {
    cudaError_t e = cudaSuccess;
    auto set = [&](const void *f) {
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(GM_SMEM - sizeof(GemmState) - 1024));
    };
    set((const void *)k_gemm<GEMM_Y, true>);
    set((const void *)k_gemm<GEMM_Y, false>);
    set((const void *)k_gemm<GEMM_GATE_UP, true>);
    set((const void *)k_gemm<GEMM_HEAD, true>);
    set((const void *)k_gemm<GEMM_HEAD, false>);
    return e;
}

}  // namespace pbd
