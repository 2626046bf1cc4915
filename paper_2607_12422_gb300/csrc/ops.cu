// ops.cu -- small kernels around the passes:
//   k_build_ids       row token ids of a draft / verify / decode pass from the device state
//   k_accept_commit   longest accepted prefix, emission, KV commit (Section 3, steps 4-5)
//   k_prefill_finish  cached lengths and first tokens after prompts
//   k_repack_tiled    row-major bf16 weights -> 128 x 64 tiles in the 128-byte swizzle layout
//   k_read_kv         paged cache -> contiguous rows (tests of the commit rule)
//   k_pack_b          adapter B rows padded to 32 columns (standalone linear)
#include "common.cuh"
#include "pbd_internal.h"

namespace pbd {

__global__ void k_pack_b(const bf16 *__restrict__ b, int N, int r, bf16 *__restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N * 32) return;
    out[i] = (i & 31) < r ? b[(size_t)(i >> 5) * r + (i & 31)] : __float2bfloat16_rn(0.f);
}

cudaError_t launch_pack_b(const void *b, int N, int r, void *out, cudaStream_t st) {
    k_pack_b<<<(N * 32 + 255) / 256, 256, 0, st>>>(static_cast<const bf16 *>(b), N, r, static_cast<bf16 *>(out));
    return cudaGetLastError();
}

// kind 0: draft rows [pending, -1 x D]; 1: verify rows [pending, d_1..d_D]; 2: decode [pending]
__global__ void k_build_ids(PassDesc pd, int kind, const int *__restrict__ pending, const int *__restrict__ drafts,
                            int D, int *__restrict__ ids) {
    const int m = blockIdx.x * blockDim.x + threadIdx.x;
    if (m >= pd.M) return;
    const int bl = m / pd.R, i = m % pd.R, b = pd.b0 + bl;
    int t;
    if (i == 0)
        t = pending[b];
    else if (kind == 0)
        t = -1;
    else
        t = drafts[bl * D + (i - 1)];
    ids[m] = t;
}

cudaError_t launch_build_ids(const PassDesc &pd, int kind, const int *pending, const int *drafts, int D, int *ids,
                             cudaStream_t st) {
    k_build_ids<<<(pd.M + 127) / 128, 128, 0, st>>>(pd, kind, pending, drafts, D, ids);
    return cudaGetLastError();
}

// Section 3, steps 4-5 on the device.  One thread per sequence.
__global__ void k_accept_commit(SeqState s, int nb, int D, const int *__restrict__ drafts,
                                const int *__restrict__ verify, const int *__restrict__ forced, int forced_stride,
                                int max_new, int out_cap, int *__restrict__ accepted_out) {
    const int b = threadIdx.x;
    const int round = *s.round;
    __syncthreads();
    if (b < nb) {
        if (s.done[b]) {
            if (accepted_out) accepted_out[b] = -1;
        } else {
            const int *d = drafts + (size_t)b * D;
            const int *v = verify + (size_t)b * (D + 1);
            int n = 0;
            while (n < D && d[n] == v[n]) ++n;
            if (forced != nullptr) n = min(max(forced[(size_t)round * forced_stride + b], 0), D);
            const int cnt = s.n_out[b];
            const int take = min(n + 1, max_new - cnt);
            for (int j = 0; j < take; ++j) s.out_tokens[(size_t)b * out_cap + cnt + j] = j < n ? d[j] : v[n];
            s.n_out[b] = cnt + take;
            s.L[b] += n + 1;
            s.pending[b] = v[n];
            if (cnt + take >= max_new) s.done[b] = 1;
            atomicAdd((unsigned long long *)&s.stats[0], 1ull);
            atomicAdd((unsigned long long *)&s.stats[1], (unsigned long long)n);
            atomicAdd((unsigned long long *)&s.stats[2], (unsigned long long)take);
            if (accepted_out) accepted_out[b] = n;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        int all = 1;
        for (int i = 0; i < nb; ++i) all &= s.done[i];
        *s.all_done = all;
        *s.round = round + 1;
    }
}

cudaError_t launch_accept_commit(const SeqState &s, int nb, int D, const int *drafts, const int *verify,
                                 const int *forced, int forced_stride, int max_new, int out_cap, int *accepted_out,
                                 cudaStream_t st) {
    const int threads = ((nb + 31) / 32) * 32;
    k_accept_commit<<<1, threads, 0, st>>>(s, nb, D, drafts, verify, forced, forced_stride, max_new, out_cap,
                                           accepted_out);
    return cudaGetLastError();
}

// Row-major [rows, K] bf16 -> 128 x 64 swizzled tiles; one 16-byte chunk per thread.  Source row
// i lands on tile row dst_row0 + (i / group) * stride + i % group (group == rows: contiguous).
__global__ void k_repack_tiled(const uint4 *__restrict__ src, int rows, int K, bf16 *__restrict__ dst, int row0,
                               int group, int stride) {
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int cpr = K / 8;
    if (idx >= (size_t)rows * cpr) return;
    const int i = (int)(idx / cpr), cg = (int)(idx % cpr);
    const int R = row0 + (i / group) * stride + (i % group);
    const int t = R >> 7, rr = R & 127, kt = cg >> 3, c = cg & 7;
    const size_t off = ((size_t)t * (K / KT) + kt) * (TILE_ROWS * KT) + rr * KT + ((c ^ (rr & 7)) << 3);
    *reinterpret_cast<uint4 *>(dst + off) = src[idx];
}

cudaError_t launch_repack_tiled_map(const void *src, int rows, int K, void *dst_tiles, int dst_row0, int group,
                                    int stride, cudaStream_t st) {
    const size_t n = (size_t)rows * (K / 8);
    k_repack_tiled<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(static_cast<const uint4 *>(src), rows, K,
                                                                static_cast<bf16 *>(dst_tiles), dst_row0, group,
                                                                stride);
    return cudaGetLastError();
}

__global__ void k_read_kv(KVCache kv, int Hkv, int d, int layer, int seq, int n, bf16 *__restrict__ k_out,
                          bf16 *__restrict__ v_out) {
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t per = (size_t)Hkv * d;
    if (idx >= (size_t)n * per) return;
    const int t = (int)(idx / per), rem = (int)(idx % per), g = rem / d, e = rem % d;
    const int page = kv.page_table[seq * kv.pages_per_seq + t / PAGE];
    const size_t off = ((((size_t)layer * kv.n_pages + page) * Hkv + g) * PAGE + (t % PAGE)) * d + e;
    k_out[idx] = static_cast<const bf16 *>(kv.k)[off];
    v_out[idx] = static_cast<const bf16 *>(kv.v)[off];
}

cudaError_t launch_read_kv(const Dims &dm, const KVCache &kv, int layer, int seq, int n, void *k_out, void *v_out,
                           cudaStream_t st) {
    const size_t total = (size_t)n * dm.Hkv * dm.d;
    if (total == 0) return cudaSuccess;
    k_read_kv<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(kv, dm.Hkv, dm.d, layer, seq, n,
                                                               static_cast<bf16 *>(k_out), static_cast<bf16 *>(v_out));
    return cudaGetLastError();
}

__global__ void k_set_len(int *L, int b, int value) { L[b] = value; }

cudaError_t launch_set_len(int *L, int b, int value, cudaStream_t st) {
    k_set_len<<<1, 1, 0, st>>>(L, b, value);
    return cudaGetLastError();
}

__global__ void k_prefill_finish(SeqState s, const RowSeg *segs, const int *ro, int n_ro, const int *first_ids,
                                 int max_new, int out_cap) {
    for (int r = threadIdx.x; r < n_ro; r += blockDim.x) {
        const RowSeg sg = segs[ro[r]];
        const int b = sg.seq, t = first_ids[r];
        s.L[b] = sg.pos0 + sg.n;
        s.pending[b] = t;
        s.out_tokens[(size_t)b * out_cap] = t;
        s.n_out[b] = 1;
        s.done[b] = max_new <= 1 ? 1 : 0;
    }
}

cudaError_t launch_prefill_finish(const SeqState &s, const RowSeg *segs, const int *ro, int n_ro, const int *first_ids,
                                  int max_new, int out_cap, cudaStream_t st) {
    k_prefill_finish<<<1, 64, 0, st>>>(s, segs, ro, n_ro, first_ids, max_new, out_cap);
    return cudaGetLastError();
}

}  // namespace pbd
