// pbd_internal.h -- host-side interface between the orchestration (pbd.cu) and the kernel
// translation units.  Plain structs of device pointers and sizes; no torch types.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "../../include/pbd.h"

namespace pbd {

typedef __nv_bfloat16 bf16;

constexpr int PAGE = 16;           // KV page length in tokens
constexpr int ATT_SPLIT = 128;     // key positions per attention split (position-aligned)
constexpr int ATT_SUBS_MAX = 2;    // partial results per split at most (its two 64-key halves)
constexpr int ATT_SPAN_MAX = 2;    // 128-key splits per attention item at most
constexpr int KT = 64;             // K elements per 128-byte swizzle atom row (bf16)
constexpr int TILE_ROWS = 128;     // output features per tensor-core tile
constexpr int TILE_BYTES = TILE_ROWS * KT * 2;  // 16 KiB per pre-tiled weight tile

enum MaskMode : int { MASK_CAUSAL = 0, MASK_BLOCK_DRAFT = 1 };

struct Dims {
    int nl, H, Hq, Hkv, d, I, V, r;
    float eps, lora_scale;
};

// One forward pass over nb sequences x R rows; row m -> sequence b0 + m / R at position L[b] + m % R.
struct PassDesc {
    int b0, nb, R, M;
    int adapter;     // LoRA delta on
    int mask_mode;   // MaskMode
    int ro_first;    // read-out rows per sequence: i in [ro_first, ro_first + ro_count)
    int ro_count;
    int nl_run;      // decoder layers the pass runs before the final norm (the draft's early exit)
    uint64_t skip = 0;  // decoder layers below nl_run the pass skips (the draft's layer skipping)
    int att_span = 1;   // consecutive 128-key splits one attention item covers (a context constant)
};

// Paged KV cache: [layer][page][Hkv][PAGE][d] bf16 for K and for V.
struct KVCache {
    void *k, *v;
    const int *page_table;  // [max_batch][pages_per_seq]
    int pages_per_seq;
    int n_pages;
};

// A weight pre-tiled for the tensor-core kernel: row tiles x k tiles of 128 x 64 bf16 in the
// 128-byte swizzle layout, 16 KiB each.  The adapter's A rows (x A^T, stacked) occupy one
// extra row tile after the main rows.
struct TiledWeight {
    const void *tiles;
    int n_main;      // main output features (multiple of 128)
    int lora_rows;   // rows of the adapter tile (r x number of adapters)
    int K;           // input features (multiple of 64)
};

// ---- persistent pass kernel (pass_kernel.cu) ----

enum MKOp : uint8_t { MK_EMBED = 0, MK_LINEAR = 1, MK_ATTN = 2, MK_FINAL = 3 };

// Timestamps per item recorded by a traced pass (%globaltimer ns; 0 = not reached):
//   0 start, 1 inputs ready, 2 work done, 3 end (next item's start);
//   linear items: 4 operand staged, 5 accumulator ready, 6 partials stored, 7 reduced,
//     8 norm scales ready (RMSNorm inputs) or act words valid (down), 9 first reduced row's
//     partial sums present, 10 its outputs computed, 11 reduction's stores issued;
//   attention items: 4 K/V pages landed, 5 V converted, 6 counted (all splits stored), 7 merged,
//     8 block pages requested, 9 q fragments loaded, 10 softmax done, 11 partials stored,
//     12 merge inputs loaded.
constexpr int MK_STAMPS = 16;

// One work item of a pass.  MK_LINEAR: lin (0 q|k|v, 1 o, 2 gate|up, 3 down), a = row tile
// (the adapter tile is the last one), b = K slice.  MK_ATTN: a = sequence in the pass, b = KV
// head, c = item index (splits c * att_span .. c * att_span + att_span - 1 of 128 keys each).
// MK_EMBED: a = row.  MK_FINAL: a = read-out index, b = row.
// Dependencies, worked out on the host: the item waits until counter wait_off (an index into the
// pass's counters, -1: none) reaches wait_tgt, and once its result is stored it adds one to each
// counter rel[k] >= 0 (a reduction, an embedded row, an attention merge).
struct __align__(16) MKItem {
    uint8_t op, lin;
    uint16_t layer;
    int32_t a, b, c;
    int32_t wait_off, wait_tgt;
    int32_t rel[2];
};

// Offsets of the pass's completion counters (ints, zeroed before every pass).
struct CounterLayout {
    int embed;      // rows embedded
    int global;     // first per-layer counter (slots before it: embed, CTAs started)
    int per_layer;  // counters per layer
    int res_o, res_dn;  // residual tiles finished after o / down
    int att;        // per (sequence, KV head): split items done (+1 once merged)
    int att_in;     // per KV head: reduced q|k|v tile slices that its attention reads
    int att_o;      // per K slice of the o projection: attention merges of the heads it reads
    int total;
};

struct MKLaunch {
    const CUtensorMap *kmap, *vmap;  // paged K / V cache, box {64 dims, 16 tokens}
    Dims dm;
    PassDesc pd;
    int grid;
    const MKItem *items;
    const int *cta_off;
    const int *nsplit;
    int *cnt;
    CounterLayout cl;
    const void *wt[4];
    size_t wt_stride[4];
    int n_main[4], lora_rows[4], K[4];
    const void *lora_b[4];
    size_t lb_stride[4];
    const void *attn_norm, *mlp_norm, *q_norm, *k_norm, *final_norm, *mask_embed, *embed_tiled;
    const float2 *rope_cs;
    int rope_rows;
    KVCache kv;
    const int *Lbuf;
    const int *ids;
    unsigned long long *part[4];  // split-K partials, tagged with the pass counter
    int *epoch;                   // pass counter (device)
    int part_rows;
    void *h, *q, *attn, *act, *x_ro;
    float *ss;
    float *o_part;
    float2 *ml_part;
    int att_splits_alloc;
    int att_subs;  // partial results per split: 2 (64-key halves) or 1 (one warp covers the 128 keys)
    int *status, *abort;
    unsigned long long *trace = nullptr;  // optional per-item timestamps
};

int mk_grid_size();
void mk_counter_layout(const Dims &dm, int max_nb, CounterLayout *cl);
void mk_build_schedule(const Dims &dm, const PassDesc &pd, const std::vector<int> &nsplit, int grid,
                       const CounterLayout &cl, std::vector<MKItem> *out, std::vector<int> *off);
size_t mk_union_bytes(int bn, int head_dim, int att_span);
int mk_slice_atoms(int lin, int K);  // 64-wide K atoms per work item of linear `lin`
cudaError_t launch_pass_kernel(const MKLaunch &L, cudaStream_t st);

// ---- decoding passes as a chain of small kernels (steps.cu) ----

struct StepArgs {
    Dims dm;
    PassDesc pd;
    const int *L, *ids;
    KVCache kv;
    bf16 *h, *q, *attn, *act;  // [rows_alloc][H], [][Hq d], [][Hq d], [][I]
    float *ss;                 // [rows_alloc][H / 128] sums of squares of h
    int rows_alloc;
    const float2 *rope_cs;
    int rope_rows;
    int att_subs;              // partial results per 128-key split
    float att_scale;
    float *o_part;             // partial results in memory: [row][head][att_splits_alloc][d],
    float2 *ml_part;           // [row][head][att_splits_alloc]
    int att_splits_alloc;
    int *status;
    int bn;                    // (set by the launcher) token columns of the MMAs
};
struct StepLin {
    const uint8_t *tiles;      // this layer's weight, pre-tiled, the adapter's rows in the last tile
    const bf16 *gain, *q_norm, *k_norm, *lora_b;  // this layer's
    int layer, K, n_main;
    int short_x;               // (host, linears 1 and 3) the activations' copies bring fewer bytes than the kernel waits for
    // set by the launcher
    CUtensorMap xmap;
    int k_tiles, katoms, ks, ring_atoms, push;
    uint32_t tmem_cols;
};
// 128-key splits of a pass's sequences end to end: sequence b has start[b] .. start[b + 1) (max_batch <= 64)
struct StepSplits {
    int start[65];
};
// whether every step of the pass fits a cluster and its shared memory (nsplit: 128-key splits of the
// longest sequence)
bool step_pass_fits(const Dims &dm, const PassDesc &pd, int subs, int nsplit);
cudaError_t launch_step_embed(const StepArgs &a, const void *embed_tiled, const void *mask_embed, cudaStream_t st);
cudaError_t launch_step_linear(int lin, StepArgs &a, StepLin &w, cudaStream_t st);
cudaError_t launch_step_attn(const StepArgs &a, const CUtensorMap &kmap, const CUtensorMap &vmap, int layer,
                             const StepSplits &sp, cudaStream_t st);
cudaError_t launch_step_final(const StepArgs &a, const void *gain, void *x_ro, cudaStream_t st);
cudaError_t configure_step_kernels();

// ---- passes over many rows: prompt processing (rows.cu, gemm.cu) ----

// Rows row0 .. row0 + n - 1 of a pass hold positions pos0 .. pos0 + n - 1 of sequence seq.
struct RowSeg {
    int row0, seq, pos0, n;
};
// One attention work item: rows_attn_tile() (row, head) pairs of a segment and KV head, from pair q0
// (pair = row in segment * heads per group + head in group).
struct RowsAttn {
    int seg, g, q0, pad;
};
struct RowsArgs {
    Dims dm;
    int M, n_seg;
    const RowSeg *segs;  // ascending row0, covering rows 0 .. M - 1
    bf16 *h, *x, *qkv, *q, *attn, *y;
    KVCache kv;
    int att_subs;        // partial results per 128-key split (as in the decoding passes)
    float att_scale;
    int max_ctas;        // CTAs per launch at most (0: no limit)
    int *status;
};
int rows_attn_tile();
cudaError_t configure_rows_kernels();
cudaError_t launch_rows_embed(const RowsArgs &a, const int *ids, const void *embed_tiled, const void *gain,
                              cudaStream_t st);
cudaError_t launch_rows_norm(const RowsArgs &a, const void *gain, cudaStream_t st);  // gain null: residual only
cudaError_t launch_rows_rope(const RowsArgs &a, int layer, const void *q_norm, const void *k_norm,
                             const float2 *rope_cs, cudaStream_t st);
cudaError_t launch_rows_attn(const RowsArgs &a, const CUtensorMap &kmap, const CUtensorMap &vmap, int layer,
                             const RowsAttn *work, int n_work, cudaStream_t st);
// x_ro[r] = final norm of the last row of segment ro[r]
cudaError_t launch_rows_final(const RowsArgs &a, const int *ro, int n_ro, const void *gain, void *x_ro, cudaStream_t st);

#ifdef __CUDACC__
// element (v, k) of a matrix in the 128 x 64 swizzled tile layout
__device__ __forceinline__ const bf16 *tiled_at(const bf16 *tiles, int K, int v, int k) {
    const int t = v >> 7, r = v & 127, kt = k >> 6, c = (k & 63) >> 3, e = k & 7;
    return tiles + ((size_t)t * (K >> 6) + kt) * (TILE_ROWS * KT) + r * KT + ((c ^ (r & 7)) << 3) + e;
}
#endif

// ---- launchers (each returns cudaGetLastError()) ----

// Standalone linear of few rows, or of few columns and a long K (linear_op.cu), one launch.  The caller fills
// everything but the last line.
struct LinOpArgs {
    CUtensorMap xmap, wmap, amap;  // boxes {64, linear_op_bn(M)}, {64, 128}, {64, r}
    int kt_per, ks, M, N, r;       // kt_per: 64-wide K atoms per slice; N: columns of y (the weight's rows, or more)
    float scale;
    const bf16 *b;
    bf16 *y;
    int vec_store;  // y is 8-byte aligned and N a multiple of 4
    int *status;
    int bn, cs, groups, stages, stage, b_off, part_off;
};
constexpr int LINEAR_OP_ROWS = 64;         // token rows of a CTA
constexpr int LINEAR_OP_MAX_CLUSTER = 16;
int linear_op_bn(int M);
double linear_op_us(int M, int N, int ks, int kt_per, int r);  // estimated time beyond an empty launch's
cudaError_t launch_linear_op(LinOpArgs &a, cudaStream_t st);
cudaError_t configure_linear_op();

// Linears of many rows (gemm.cu).  The caller fills everything but the last line.
enum GemmMode { GEMM_Y = 0, GEMM_GATE_UP = 1, GEMM_HEAD = 2 };
struct GemmArgs {
    CUtensorMap xmap;        // token rows, box {64, bn}
    CUtensorMap wmap;        // row-major weight, box {64, 128} (when wt is null)
    CUtensorMap bmap, umap;  // adapter (delta): B rows, box {64, 128}; u rows, box {64, bn}
    const uint8_t *wt;       // pre-tiled weight (GEMM_GATE_UP: gate and up interleaved in 64-row blocks)
    int k_tiles, slice_atoms, n_slices;  // 64-wide K atoms; atoms per slice; slices
    int f_tiles;             // 128-feature tiles (GEMM_GATE_UP: of act features)
    int bn, M;               // token tile (a multiple of 16, at most 256; 128 for GEMM_GATE_UP), token rows
    int rows;                // features stored (the vocabulary for GEMM_HEAD)
    int delta;               // adapter on: y += scale * u B^T
    float scale;
    bf16 *y;                 // [M][ld]
    int ld, vec_store;       // vec_store: y is 16-byte aligned and ld a multiple of 8
    float *logits;           // GEMM_HEAD: [M][rows] or null
    float *tile_max;         // GEMM_HEAD: per CTA and token the (max, lowest argmax), [grid][M]
    int *tile_arg;
    int *status;
    int m_tiles, stages, stage_atoms;
};
// ctas: CTAs at most (0: one per SM)
cudaError_t launch_gemm(GemmMode mode, GemmArgs &a, int ctas, cudaStream_t st);
int gemm_pick_bn(int M, int f_tiles, int k_tiles, int max_bn, int ctas);
double gemm_us(int M, int f_tiles, int k_tiles, int bn);  // estimated time of a GEMM_Y launch beyond an empty one's
int gemm_ctas();  // CTAs of a launch with ctas = 0
cudaError_t configure_gemm_kernels();

// lm_head over M <= 256 read-out rows: per CTA the (max, lowest argmax) of each row ([*n_parts][M]
// entries of tile_max / tile_arg, at most V / 128 of them), and optionally the fp32 logits [M][V].
// x_map: box {64, lm_head_box(M, K)}.  The weight is w.tiles (pre-tiled) or, when that is null, the
// row-major matrix behind w_map.
int lm_head_box(int M, int K);
cudaError_t launch_lm_head(const CUtensorMap &x_map, const TiledWeight &w, const CUtensorMap *w_map, int M,
                           float *tile_max, int *tile_arg, int *n_parts, float *logits, int *status, cudaStream_t st);

cudaError_t launch_argmax_reduce(const float *tile_max, const int *tile_arg, int n_parts, int rows, int *ids_out,
                                 cudaStream_t st);

// Builds the row token ids of a pass from the device state: draft [pending, -1 x D],
// verify [pending, drafts], decode [pending].
cudaError_t launch_build_ids(const PassDesc &pd, int kind, const int *pending, const int *drafts, int D, int *ids,
                             cudaStream_t st);

struct SeqState {
    int *L;          // [B] committed length
    int *pending;    // [B]
    int *n_out;      // [B]
    int *done;       // [B]
    int *all_done;   // [1]
    int *out_tokens; // [B][max_new_cap]
    int *round;      // [1] rounds executed (index into the forced-n sequence)
    long long *stats;// [3]: rounds, accepted, emitted
};

// Accept/commit for nb sequences: n from drafts vs verify ids (or forced), emit, advance.
cudaError_t launch_accept_commit(const SeqState &s, int nb, int D, const int *drafts, const int *verify,
                                 const int *forced, int forced_stride, int max_new, int out_cap,
                                 int *accepted_out, cudaStream_t st);

// Repack rows [0, rows) of a row-major bf16 matrix [rows, K] into the tiled layout: source row i
// on tile row dst_row0 + (i / group) * stride + i % group (gate and up rows interleaved in 64-row
// blocks inside each 128-row tile; group = rows: contiguous).
cudaError_t launch_repack_tiled_map(const void *src, int rows, int K, void *dst_tiles, int dst_row0, int group,
                                    int stride, cudaStream_t st);

cudaError_t launch_read_kv(const Dims &dm, const KVCache &kv, int layer, int seq, int n, void *k_out, void *v_out,
                           cudaStream_t st);

// L[b] = value.
cudaError_t launch_set_len(int *L, int b, int value, cudaStream_t st);

// After the prompts that end in segments ro[0 .. n_ro): L = the segment's end, pending = first token
// first_ids[r] = output token 0.
cudaError_t launch_prefill_finish(const SeqState &s, const RowSeg *segs, const int *ro, int n_ro, const int *first_ids,
                                  int max_new, int out_cap, cudaStream_t st);

// B [N, r] -> [N, 32], zero beyond r (standalone linear of many rows whose B has no TMA layout).
cudaError_t launch_pack_b(const void *b, int N, int r, void *out, cudaStream_t st);

// 2-D bf16 row-major [rows, cols] tensor map, rows ld values apart (0: cols), box {64, box_rows}, 128-byte swizzle.
bool encode_bf16_map(CUtensorMap *map, const void *base, int rows, int cols, int box_rows, int ld = 0);

// Per-instantiation kernel attributes (dynamic shared memory), set once before any capture.
cudaError_t configure_linear_kernels();

// The standalone linear shared by pbd_op_linear and pbd_op_linear_static: scratch is at least
// 1024 bytes for the status word, `tiles` (N / 128 (+ 1 with an adapter)) * (K / 64) * 16 KiB and
// `part` 4 * slices * M * (N + r) bytes, all 1024-byte aligned, tiles right behind the first 1024.
struct LinearScratch {
    uint8_t *status, *tiles, *part;
};
pbd_status run_linear_op(int M, int K, int N, int r, float scale, const void *d_x, const void *d_w, const void *d_a,
                         const void *d_b, void *d_y, const LinearScratch &ws, cudaStream_t st, const char *who);

// Records the message pbd_op_last_error() returns on this thread.
void op_record_error(const char *msg);

// Single-op status words: wait for the stream and read the latched DEV_* code; turn a nonzero
// code into PBD_ERR_DEVICE with its message (pbd_op_last_error()).
pbd_status read_device_code(const int *d_status, cudaStream_t st, int *code, const char *who);
pbd_status device_fail(int code, const char *who);

}  // namespace pbd
