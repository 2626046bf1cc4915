// ops_api.cu -- single-kernel C entry points (include/pbd_ops.h) and the TMA descriptor helper
// shared with the context code.  The linear and the lm_head read the caller's row-major weights
// through tensor maps and sum over K in the same slices and order as the decoder passes.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdio>
#include <string>

#include "../../include/pbd_ops.h"
#include "common.cuh"
#include "pbd_internal.h"

namespace pbd {

typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// 2-D bf16 row-major [rows, cols] tensor map with box {64, box_rows}, 128-byte swizzle; rows lie ld values apart
// (0: cols).
bool encode_bf16_map(CUtensorMap *map, const void *base, int rows, int cols, int box_rows, int ld) {
    static EncodeTiledFn enc = nullptr;
    if (!enc) {
        void *fn = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) !=
                cudaSuccess ||
            fn == nullptr || q != cudaDriverEntryPointSuccess)
            return false;
        enc = reinterpret_cast<EncodeTiledFn>(fn);
    }
    if (ld == 0) ld = cols;
    if ((reinterpret_cast<uintptr_t>(base) & 15) || (ld * 2) % 16) return false;
    cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
    cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
    cuuint32_t box[2] = {(cuuint32_t)KT, (cuuint32_t)box_rows};
    cuuint32_t es[2] = {1, 1};
    return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(base), dims, strides, box, es,
               CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace pbd

using namespace pbd;

namespace {

thread_local std::string g_op_err;

pbd_status op_fail(pbd_status s, const char *msg, cudaError_t e = cudaSuccess) {
    char b[256];
    snprintf(b, sizeof b, "%s%s%s", msg, e != cudaSuccess ? ": " : "", e != cudaSuccess ? cudaGetErrorString(e) : "");
    g_op_err = b;
    return s;
}

struct LinearPlan {
    size_t tiles_off, part_off, status_off, total;
    int k_splits, row_tiles;
};

bool plan_linear(int M, int K, int N, int r, LinearPlan *p) {
    if (M < 1 || M > 4096 || K < 64 || K % 64 || N < 128 || N % 128 || r < 0 || r > 32) return false;
    const int kt = K / KT;
    p->k_splits = (kt % 4 == 0) ? kt / 4 : 1;
    p->row_tiles = N / TILE_ROWS + (r > 0 ? 1 : 0);
    size_t off = 0;
    auto take = [&](size_t bytes) {
        off = (off + 1023) / 1024 * 1024;
        const size_t o = off;
        off += bytes;
        return o;
    };
    p->status_off = take(256);
    p->tiles_off = take((size_t)p->row_tiles * kt * TILE_BYTES);
    p->part_off = take(sizeof(float) * (size_t)p->k_splits * M * (N + r));
    p->total = off;
    return true;
}

}  // namespace

namespace pbd {

// Waits for d_stream, then reads the status word a kernel may have latched (a DEV_* code).  The copy goes behind the
// work instead of following a wait for it: one round trip to the device (after an empty kernel 14.6 us
// against 18.8).
pbd_status read_device_code(const int *d_status, cudaStream_t st, int *code, const char *who) {
    cudaError_t e = cudaMemcpyAsync(code, d_status, sizeof(int), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) {
        char b[128];
        snprintf(b, sizeof b, "%s: reading the status word", who);
        return op_fail(PBD_ERR_CUDA, b, e);
    }
    return PBD_OK;
}

// whether [a, a + na) and [b, b + nb) share a byte
static bool overlap(const void *a, size_t na, const void *b, size_t nb) {
    const uintptr_t x = reinterpret_cast<uintptr_t>(a), y = reinterpret_cast<uintptr_t>(b);
    return x < y + nb && y < x + na;
}

// linear_op.cu, one launch that spreads the K slices over CTAs, or gemm.cu, whose CTAs keep whole tiles' sums in registers
// and take all of K: up to 64 rows and 16 slices the first, beyond that the one with the shorter estimated
// time.  Both ways, us per call with cold caches, rank 0 (and with re-tiling and split-K partial sums in
// memory): M = 17, K = 16384, N = 128: 22 and 62 (28); M = 100, K = 4096, N = 128: 14 and 22 (26); M = 64,
// K = 16384, N = 4096: 92 and 65 (127); M = 400, K = 3072, N = 1024: 31 and 19 (43).  With gemm.cu the adapter's
// u = bf16(x A^T) comes first, one tile of features by either kernel (the whole of K in one CTA per 64 rows, or
// spread: M = 100, K = 16384: 59 and 22 us), and enters the tile as one more MMA group.
pbd_status run_linear_op(int M, int K, int N, int r, float scale, const void *d_x, const void *d_w, const void *d_a,
                         const void *d_b, void *d_y, const LinearScratch &ws, cudaStream_t st, const char *who) {
    const size_t y_bytes = (size_t)M * N * 2;
    if (overlap(d_y, y_bytes, d_x, (size_t)M * K * 2) || overlap(d_y, y_bytes, d_w, (size_t)N * K * 2) ||
        (r > 0 && (overlap(d_y, y_bytes, d_a, (size_t)r * K * 2) || overlap(d_y, y_bytes, d_b, (size_t)N * r * 2)))) {
        // The operands are read where they lie, by some CTAs after others have stored: y goes through the scratch.
        // Of part's 4 M N bytes or more u takes the first 64 M (N is at least 128), y the second 2 M N.
        uint8_t *y = ws.part + y_bytes;
        const pbd_status s = run_linear_op(M, K, N, r, scale, d_x, d_w, d_a, d_b, y, ws, st, who);
        if (s != PBD_OK) return s;
        const cudaError_t e = cudaMemcpyAsync(d_y, y, y_bytes, cudaMemcpyDeviceToDevice, st);
        return e == cudaSuccess ? PBD_OK : op_fail(PBD_ERR_CUDA, "copying an output that lies over an operand", e);
    }
    auto bad = [&](pbd_status s, const char *what, cudaError_t e = cudaSuccess) {
        char b[160];
        snprintf(b, sizeof b, "%s: %s", who, what);
        return op_fail(s, b, e);
    };
    const int kt = K / KT, ks = kt % 4 == 0 ? kt / 4 : 1, f_tiles = N / TILE_ROWS;
    int *status = reinterpret_cast<int *>(ws.status);
    cudaError_t e;
    if ((e = configure_linear_kernels()) != cudaSuccess) return bad(PBD_ERR_CUDA, "configure", e);
    // y[M][ld] = x w^T (+ the delta of rank ra) for the `rows` rows of w
    auto op = [&](const void *w, int rows, int ld, int ra, void *y) {
        LinOpArgs a{};
        if (!encode_bf16_map(&a.xmap, d_x, M, K, linear_op_bn(M))) return bad(PBD_ERR_INVALID_ARG, "x not TMA-mappable");
        if (!encode_bf16_map(&a.wmap, w, rows, K, TILE_ROWS))
            return bad(PBD_ERR_INVALID_ARG, w == d_w ? "W not TMA-mappable" : "A not TMA-mappable");
        a.amap = a.wmap;
        if (ra > 0 && !encode_bf16_map(&a.amap, d_a, ra, K, ra)) return bad(PBD_ERR_INVALID_ARG, "A not TMA-mappable");
        a.kt_per = kt / ks;
        a.ks = ks;
        a.M = M;
        a.N = ld;
        a.r = ra;
        a.scale = scale;
        a.b = static_cast<const bf16 *>(d_b);
        a.y = static_cast<bf16 *>(y);
        a.vec_store = (reinterpret_cast<uintptr_t>(y) & 7) == 0;
        a.status = status;
        const cudaError_t err = launch_linear_op(a, st);
        return err == cudaSuccess ? PBD_OK : bad(PBD_ERR_CUDA, "linear", err);
    };
    const int bn = gemm_pick_bn(M, f_tiles, kt, 256, gemm_ctas());
    const double u_gemm = gemm_us(M, 1, kt, 64), u_op = linear_op_us(M, 32, ks, kt / ks, 0) + 1.0;  // (+ a full launch)
    if ((M <= LINEAR_OP_ROWS && ks <= LINEAR_OP_MAX_CLUSTER) ||
        linear_op_us(M, N, ks, kt / ks, r) < gemm_us(M, f_tiles, kt, bn) + (r > 0 ? std::min(u_gemm, u_op) : 0.0)) {
        if ((e = cudaMemsetAsync(status, 0, 256, st)) != cudaSuccess) return bad(PBD_ERR_CUDA, "memset", e);
        return op(d_w, N, N, r, d_y);
    }
    GemmArgs a{};
    a.bn = bn;
    if (!encode_bf16_map(&a.xmap, d_x, M, K, a.bn)) return bad(PBD_ERR_INVALID_ARG, "x not TMA-mappable");
    if (!encode_bf16_map(&a.wmap, d_w, N, K, TILE_ROWS)) return bad(PBD_ERR_INVALID_ARG, "W not TMA-mappable");
    a.k_tiles = kt;
    a.slice_atoms = kt / ks;
    a.n_slices = ks;
    a.f_tiles = f_tiles;
    a.M = M;
    a.rows = N;
    a.scale = scale;
    a.y = static_cast<bf16 *>(d_y);
    a.ld = N;
    a.vec_store = (reinterpret_cast<uintptr_t>(d_y) & 15) == 0;
    a.status = status;
    if ((e = cudaMemsetAsync(status, 0, 256, st)) != cudaSuccess) return bad(PBD_ERR_CUDA, "memset", e);
    if (r > 0) {
        // u [M][32] and a padded B [N][32].  Each fits its area whatever the sizes: `part` holds at least 512 bytes a row,
        // `tiles` 128 a column.  (Behind u, B would not: `part` is small for few rows.)
        uint8_t *u = ws.part, *bp = ws.tiles;
        if (u_op < u_gemm) {
            const pbd_status s = op(d_a, r, 32, 0, u);
            if (s != PBD_OK) return s;
        } else {
            GemmArgs g = a;
            g.bn = 64;
            if (!encode_bf16_map(&g.xmap, d_x, M, K, g.bn)) return bad(PBD_ERR_INVALID_ARG, "x not TMA-mappable");
            if (!encode_bf16_map(&g.wmap, d_a, r, K, TILE_ROWS)) return bad(PBD_ERR_INVALID_ARG, "A not TMA-mappable");
            g.f_tiles = 1;
            g.rows = 32;
            g.y = reinterpret_cast<bf16 *>(u);
            g.ld = 32;
            g.vec_store = 1;
            if ((e = launch_gemm(GEMM_Y, g, 0, st)) != cudaSuccess) return bad(PBD_ERR_CUDA, "adapter rows", e);
        }
        a.delta = 1;
        // (r columns: the rest arrive as zeros.  What the kernel computed there, 0 x, is NaN where x is infinite.)
        bool ok = encode_bf16_map(&a.umap, u, M, r, a.bn, 32);
        if (r % 8 == 0 && (reinterpret_cast<uintptr_t>(d_b) & 15) == 0) {
            ok = ok && encode_bf16_map(&a.bmap, d_b, N, r, TILE_ROWS);
        } else {  // no TMA layout: rows padded to 32
            if ((e = launch_pack_b(d_b, N, r, bp, st)) != cudaSuccess) return bad(PBD_ERR_CUDA, "pack B", e);
            ok = ok && encode_bf16_map(&a.bmap, bp, N, 32, TILE_ROWS);
        }
        if (!ok) return bad(PBD_ERR_CUDA, "tensor map encode failed");
    }
    if ((e = launch_gemm(GEMM_Y, a, 0, st)) != cudaSuccess) return bad(PBD_ERR_CUDA, "linear", e);
    return PBD_OK;
}

const char *device_code_name(int code) {
    switch (code) {
        case DEV_TIMEOUT_LOAD: return "a weight or operand copy never completed";
        case DEV_TIMEOUT_MMA: return "a tensor-core accumulation never completed";
        case DEV_TIMEOUT_SLOT: return "a shared-memory ring slot was never released";
        case DEV_BAD_TOKEN: return "token id outside the vocabulary";
        case DEV_BAD_POSITION: return "position beyond the reserved KV pages";
        case DEV_TIMEOUT_DEP: return "a work item's inputs never completed";
        default: return "unknown device code";
    }
}

pbd_status device_fail(int code, const char *who) {
    char b[256];
    snprintf(b, sizeof b, "%s: device status %d latched by a kernel (%s); the outputs of that call are invalid", who,
             code, device_code_name(code));
    g_op_err = b;
    return PBD_ERR_DEVICE;
}

}  // namespace pbd

extern "C" {

size_t pbd_op_linear_workspace_bytes(int32_t M, int32_t K, int32_t N, int32_t r) {
    LinearPlan p;
    return plan_linear(M, K, N, r, &p) ? p.total : 0;
}

pbd_status pbd_op_linear(int32_t M, int32_t K, int32_t N, int32_t r, float scale, const void *d_x, const void *d_w,
                         const void *d_a, const void *d_b, void *d_y, void *d_ws, size_t ws_bytes, void *d_stream) {
    const bool lora = r > 0 && d_a != nullptr && d_b != nullptr;
    const int rr = lora ? r : 0;
    LinearPlan p;
    if (!plan_linear(M, K, N, rr, &p)) return op_fail(PBD_ERR_INVALID_ARG, "pbd_op_linear: unsupported sizes");
    if (!d_x || !d_w || !d_y) return op_fail(PBD_ERR_INVALID_ARG, "pbd_op_linear: null pointer");
    if (!d_ws || (reinterpret_cast<uintptr_t>(d_ws) & 1023) || ws_bytes < p.total)
        return op_fail(PBD_ERR_WORKSPACE, "pbd_op_linear: workspace missing, misaligned or too small");
    uint8_t *ws = static_cast<uint8_t *>(d_ws);
    return run_linear_op(M, K, N, rr, scale, d_x, d_w, d_a, d_b, d_y,
                         LinearScratch{ws + p.status_off, ws + p.tiles_off, ws + p.part_off},
                         static_cast<cudaStream_t>(d_stream), "pbd_op_linear");
}

size_t pbd_op_lm_head_workspace_bytes(int32_t M, int32_t H, int32_t V) {
    if (M < 1 || M > 256 || H < 64 || H % 64 || V < 128 || V % 128) return 0;
    size_t tiles = (size_t)(V / TILE_ROWS) * (H / KT) * TILE_BYTES;
    size_t red = (size_t)(V / TILE_ROWS) * M * 8;
    return 1024 + (tiles + 1023) / 1024 * 1024 + (red + 1023) / 1024 * 1024;
}

pbd_status pbd_op_lm_head_argmax(int32_t M, int32_t H, int32_t V, const void *d_x, const void *d_embed,
                                 int32_t *d_ids, float *d_logits_opt, void *d_ws, size_t ws_bytes, void *d_stream) {
    const size_t need = pbd_op_lm_head_workspace_bytes(M, H, V);
    if (need == 0) return op_fail(PBD_ERR_INVALID_ARG, "pbd_op_lm_head_argmax: unsupported sizes");
    if (!d_x || !d_embed || !d_ids) return op_fail(PBD_ERR_INVALID_ARG, "pbd_op_lm_head_argmax: null pointer");
    if (!d_ws || (reinterpret_cast<uintptr_t>(d_ws) & 1023) || ws_bytes < need)
        return op_fail(PBD_ERR_WORKSPACE, "pbd_op_lm_head_argmax: workspace missing, misaligned or too small");
    cudaStream_t st = static_cast<cudaStream_t>(d_stream);
    uint8_t *ws = static_cast<uint8_t *>(d_ws);
    int *status = reinterpret_cast<int *>(ws);
    const size_t tiles_bytes = (size_t)(V / TILE_ROWS) * (H / KT) * TILE_BYTES;
    if (d_logits_opt && overlap(d_logits_opt, sizeof(float) * (size_t)M * V, d_embed, (size_t)V * H * 2)) {
        // logits over the table that is read while they are stored: the table is read from a copy
        const cudaError_t e = cudaMemcpyAsync(ws + 1024, d_embed, (size_t)V * H * 2, cudaMemcpyDeviceToDevice, st);
        if (e != cudaSuccess) return op_fail(PBD_ERR_CUDA, "pbd_op_lm_head_argmax: copying the table", e);
        d_embed = ws + 1024;
    }
    TiledWeight w;
    w.tiles = nullptr;  // read through w_map
    w.n_main = V;
    w.lora_rows = 0;
    w.K = H;
    float *tmax = reinterpret_cast<float *>(ws + 1024 + (tiles_bytes + 1023) / 1024 * 1024);
    int *targ = reinterpret_cast<int *>(tmax + (size_t)(V / TILE_ROWS) * M);
    CUtensorMap map, w_map;
    if (!encode_bf16_map(&map, d_x, M, H, lm_head_box(M, H)))
        return op_fail(PBD_ERR_INVALID_ARG, "pbd_op_lm_head_argmax: x not TMA-mappable");
    if (!encode_bf16_map(&w_map, d_embed, V, H, TILE_ROWS))
        return op_fail(PBD_ERR_INVALID_ARG, "pbd_op_lm_head_argmax: embed not TMA-mappable");
    cudaError_t e;
    int n_parts = 0;
    if ((e = configure_linear_kernels()) != cudaSuccess) return op_fail(PBD_ERR_CUDA, "configure", e);
    if ((e = cudaMemsetAsync(status, 0, 256, st)) != cudaSuccess) return op_fail(PBD_ERR_CUDA, "memset", e);
    if ((e = launch_lm_head(map, w, &w_map, M, tmax, targ, &n_parts, d_logits_opt, status, st)) != cudaSuccess)
        return op_fail(PBD_ERR_CUDA, "lm_head", e);
    if ((e = launch_argmax_reduce(tmax, targ, n_parts, M, d_ids, st)) != cudaSuccess)
        return op_fail(PBD_ERR_CUDA, "argmax", e);
    return PBD_OK;
}

pbd_status pbd_op_status(const void *d_ws, void *d_stream, int32_t *h_device_code) {
    if (h_device_code) *h_device_code = 0;
    if (!d_ws || (reinterpret_cast<uintptr_t>(d_ws) & 1023))
        return op_fail(PBD_ERR_INVALID_ARG, "pbd_op_status: workspace missing or misaligned");
    int code = 0;
    pbd_status s = read_device_code(static_cast<const int *>(d_ws), static_cast<cudaStream_t>(d_stream), &code,
                                    "pbd_op_status");
    if (s != PBD_OK) return s;
    if (h_device_code) *h_device_code = code;
    return code == 0 ? PBD_OK : device_fail(code, "pbd_op_status");
}

const char *pbd_op_last_error(void) { return g_op_err.c_str(); }

}  // extern "C"

namespace pbd {
void op_record_error(const char *msg) { g_op_err = msg; }
}  // namespace pbd
