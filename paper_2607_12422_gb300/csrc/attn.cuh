// attn.cuh -- tensor-core steps of the attention, shared by the pass kernel and the many-row kernel (their
// results must agree bit for bit).
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

// O += P V over 16 keys; vaddr: shared address of the first key's row plus attn_v_lane.  ma, mb: masks
// of the fragment registers (keys 2 tq, 2 tq + 1 and + 8, + 9).
template <int DH>
__device__ __forceinline__ void attn_pv(uint32_t vaddr, const uint32_t (&pa)[4], uint32_t ma, uint32_t mb,
                                        float (&oc)[DH / 8][4]) {
#pragma unroll
    for (int dt = 0; dt < DH / 8; dt += 2) {
        const uint32_t va = (vaddr ^ ((dt & 7) << 4)) + (dt >> 3) * ATT_SUB_BYTES;
        uint32_t r0, r1, r2, r3;
        asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                     : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                     : "r"(va));
        mma_m16n8k16_bf16(oc[dt], pa, r0 & ma, r1 & mb);
        mma_m16n8k16_bf16(oc[dt + 1], pa, r2 & ma, r3 & mb);
    }
}

}  // namespace pbd
