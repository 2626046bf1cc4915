// attn.cuh -- tensor-core steps of the attention, shared by the pass kernel and the decoding chain (their
// results must agree bit for bit, and with rows.cu's).
//
// Staged K and V: DH / 64 sub-tiles of [128 keys x 128 bytes] in the 128-byte swizzle layout (16-byte
// chunk c of key n at (c ^ (n & 7)) * 16), as the tiled TMA writes them, 1024-byte aligned.  The key
// rows that a lane addresses are congruent to lane % 8 modulo 8, so the swizzle is a constant of the
// lane: addresses are the lane's base, XOR a constant of the chunk, plus immediates.
#pragma once

#include "common.cuh"
#include "pbd_internal.h"

namespace pbd {

constexpr int ATT_SUB_BYTES = ATT_SPLIT * 128;

// the lane's offset for K fragments (ldmatrix.x4: matrix lane / 8 holds 8 dims of the keys) ...
__device__ __forceinline__ uint32_t attn_k_lane(int lane) {
    return (uint32_t)((lane & 7) * 128 + (((lane >> 3) ^ (lane & 7)) << 4));
}
// ... and for V fragments (transposed: matrices 0, 1 keys 0-7, 8-15 of 8 dims, 2, 3 of the next 8)
__device__ __forceinline__ uint32_t attn_v_lane(int lane) {
    return (uint32_t)(((lane & 7) + ((lane >> 3) & 1) * 8) * 128 + (((lane >> 4) ^ (lane & 7)) << 4));
}

// Raw scores of one 16-row query tile against 32 keys; kaddr: shared address of the first key's row plus
// attn_k_lane.  Each score accumulates over the head's dims in order; the four 8-key tiles take turns,
// so that four chains of dependent MMAs are in flight.
template <int DH>
__device__ __forceinline__ void attn_scores(uint32_t kaddr, const uint32_t (&qa)[DH / 16][4], float (&sc)[4][4]) {
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) sc[nt][0] = sc[nt][1] = sc[nt][2] = sc[nt][3] = 0.f;
#pragma unroll
    for (int ks = 0; ks < DH / 16; ks += 2) {
        const uint32_t ka = (kaddr ^ ((ks & 2) << 5)) + (ks >> 2) * ATT_SUB_BYTES;
        uint32_t b[4][4];
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
            asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                         : "=r"(b[nt][0]), "=r"(b[nt][1]), "=r"(b[nt][2]), "=r"(b[nt][3])
                         : "r"(ka + nt * 1024));
#pragma unroll
        for (int e = 0; e < 2; ++e)
#pragma unroll
            for (int nt = 0; nt < 4; ++nt) mma_m16n8k16_bf16(sc[nt], qa[ks + e], b[nt][2 * e], b[nt][2 * e + 1]);
    }
}

// The same with the query tile in shared memory, 16 rows of ATT_Q_PITCH bytes (16 of padding: the eight rows of
// a fragment fall on distinct banks); qaddr: its address plus attn_q_lane.  Saves the fragments' registers.
__host__ __device__ constexpr int ATT_Q_PITCH(int dh) { return 2 * dh + 16; }
template <int DH>
__device__ __forceinline__ uint32_t attn_q_lane(int lane) {
    return (uint32_t)(((lane & 7) + ((lane >> 3) & 1) * 8) * ATT_Q_PITCH(DH) + (lane >> 4) * 16);
}
template <int DH>
__device__ __forceinline__ void attn_scores_sq(uint32_t kaddr, uint32_t qaddr, float (&sc)[4][4]) {
#pragma unroll
    for (int nt = 0; nt < 4; ++nt) sc[nt][0] = sc[nt][1] = sc[nt][2] = sc[nt][3] = 0.f;
#pragma unroll
    for (int ks = 0; ks < DH / 16; ks += 2) {
        const uint32_t ka = (kaddr ^ ((ks & 2) << 5)) + (ks >> 2) * ATT_SUB_BYTES;
        uint32_t b[4][4], qa[2][4];
#pragma unroll
        for (int e = 0; e < 2; ++e)
            asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                         : "=r"(qa[e][0]), "=r"(qa[e][1]), "=r"(qa[e][2]), "=r"(qa[e][3])
                         : "r"(qaddr + (ks + e) * 32));
#pragma unroll
        for (int nt = 0; nt < 4; ++nt)
            asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                         : "=r"(b[nt][0]), "=r"(b[nt][1]), "=r"(b[nt][2]), "=r"(b[nt][3])
                         : "r"(ka + nt * 1024));
#pragma unroll
        for (int e = 0; e < 2; ++e)
#pragma unroll
            for (int nt = 0; nt < 4; ++nt) mma_m16n8k16_bf16(sc[nt], qa[e], b[nt][2 * e], b[nt][2 * e + 1]);
    }
}

// O += P V over 16 keys; vaddr: shared address of the first key's row plus attn_v_lane.  ma, mb: masks
// of the fragment registers (keys 2 tq, 2 tq + 1 and + 8, + 9).
template <int DH>
__device__ __forceinline__ void attn_pv(uint32_t vaddr, const uint32_t (&pa)[4], uint32_t ma, uint32_t mb,
                                        float (&oc)[DH / 8][4]) {
    // four fragments on their way before the first is used
#pragma unroll
    for (int d0 = 0; d0 < DH / 8; d0 += 8) {
        uint32_t r[4][4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t va = (vaddr ^ ((2 * i) << 4)) + (d0 >> 3) * ATT_SUB_BYTES;
            asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                         : "=r"(r[i][0]), "=r"(r[i][1]), "=r"(r[i][2]), "=r"(r[i][3])
                         : "r"(va));
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            mma_m16n8k16_bf16(oc[d0 + 2 * i], pa, r[i][0] & ma, r[i][1] & mb);
            mma_m16n8k16_bf16(oc[d0 + 2 * i + 1], pa, r[i][2] & ma, r[i][3] & mb);
        }
    }
}

}  // namespace pbd
