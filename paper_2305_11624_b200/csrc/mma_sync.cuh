// Warp-level tensor-core helpers (mma.sync / ldmatrix) for the problems whose N dimension is too narrow
// for a 128-row tcgen05 tile.
#pragma once
#include <cstdint>

namespace convbn {

// D (16 x 8, fp32) += A (16 x 16, bf16, row-major fragments) x B (16 x 8, bf16, column fragments).
// Lane (g = lane / 4, t = lane % 4): a0 = A[g][2t..2t+1], a1 = A[g+8][2t..], a2 = A[g][2t+8..], a3 = A[g+8][2t+8..];
// b0 = B[2t..2t+1][g], b1 = B[2t+8..2t+9][g]; c0, c1 = D[g][2t, 2t+1], c2, c3 = D[g+8][2t, 2t+1].
__device__ __forceinline__ void mma_16x8x16_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                                 uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// The same with IEEE-half operands, and the choice between the two at compile time.
__device__ __forceinline__ void mma_16x8x16_f16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                                uint32_t b0, uint32_t b1) {
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
template <bool H>
__device__ __forceinline__ void mma_16x8x16_t(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                              uint32_t b0, uint32_t b1) {
    if constexpr (H) mma_16x8x16_f16(c, a0, a1, a2, a3, b0, b1);
    else mma_16x8x16_bf16(c, a0, a1, a2, a3, b0, b1);
}

// Four 8 x 8 bf16 matrices from shared memory: lanes 8i..8i+7 give the 16-byte row addresses of matrix i;
// register i of every lane receives its two elements of matrix i in MMA fragment order.
__device__ __forceinline__ void ldmatrix_x4(uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3, uint32_t smem_addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(smem_addr)
                 : "memory");
}

// The reverse: register i of lane (g, t) holds elements [row g][columns 2t, 2t + 1] of matrix i; lanes 8i..8i+7 give
// the addresses of its 16-byte rows.
__device__ __forceinline__ void stmatrix_x4(uint32_t smem_addr, uint32_t r0, uint32_t r1, uint32_t r2, uint32_t r3) {
    asm volatile("stmatrix.sync.aligned.m8n8.x4.shared.b16 [%0], {%1, %2, %3, %4};"
                 ::"r"(smem_addr), "r"(r0), "r"(r1), "r"(r2), "r"(r3)
                 : "memory");
}

// ldmatrix with every matrix transposed on the way: register i of lane (g, t) receives elements
// [row 2t][column g] and [row 2t + 1][column g] of matrix i.
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3,
                                                  uint32_t smem_addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(smem_addr)
                 : "memory");
}
// Two transposed matrices (row addresses from lanes 0-7 and 8-15).
__device__ __forceinline__ void ldmatrix_x2_trans(uint32_t &r0, uint32_t &r1, uint32_t smem_addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0, %1}, [%2];"
                 : "=r"(r0), "=r"(r1)
                 : "r"(smem_addr)
                 : "memory");
}

}  // namespace convbn
