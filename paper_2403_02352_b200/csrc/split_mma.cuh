// 64 x 64 x 64 products of fp32 tiles on the tensor cores (mma.sync m16n8k16) with both operands cut into two fp16 parts:
// x s = hi + lo + (at most 2^-23 |x s| or 2^-25, whichever is larger), s a power of two that brings the operand into
// fp16's range, product = lo hi + hi lo + hi hi (the lo lo term is below 2^-22). The parts are cut once, when a tile goes
// to shared memory, and read with ldmatrix. Against the same product from TF32 parts (m16n8k8, operands cut in registers by
// every warp that reads them): half the MMA instructions, a quarter of the shared-memory loads and no cutting in the
// loop: 2240 -> 950 cycles per product and CTA of 256 threads, and one bit more in each part.
#pragma once
#include "common.cuh"
#include <cuda_fp16.h>

namespace hs {

constexpr int LDH = 72;                       // row stride (halves): rows 36 banks apart, ldmatrix is conflict-free
constexpr int PLANE = 64 * LDH;               // halves of one part of a tile
constexpr size_t TILE_BYTES = 2 * PLANE * sizeof(__half);

// four values, already scaled, as two fp16 parts at (row, c .. c + 3) of a tile
__device__ __forceinline__ void put4(__half *tile, int row, int c, float4 v)
{
    const __half2 h0 = __floats2half2_rn(v.x, v.y), h1 = __floats2half2_rn(v.z, v.w);
    const float2 f0 = __half22float2(h0), f1 = __half22float2(h1);
    const __half2 l0 = __floats2half2_rn(v.x - f0.x, v.y - f0.y), l1 = __floats2half2_rn(v.z - f1.x, v.w - f1.y);
    *(uint2 *)(tile + row * LDH + c) = make_uint2(*(const uint32_t *)&h0, *(const uint32_t *)&h1);
    *(uint2 *)(tile + PLANE + row * LDH + c) = make_uint2(*(const uint32_t *)&l0, *(const uint32_t *)&l1);
}

template <bool TRANS> __device__ __forceinline__ void ldsm4(uint32_t addr, uint32_t (&r)[4])
{
    if (TRANS) asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                            : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
    else asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void mma_f16(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1)
{
    asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// acc (this warp's 16 x 32 part of the result: rows m0 .., columns n0 ..) += A B. A_T: A[m][k] = At[k][m], otherwise
// At[m][k]; B_T: B[k][n] = Bt[n][k], otherwise Bt[k][n]. Thread: rows m0 + g, + 8, columns n0 + 8 nt + 2 t, + 1.
template <bool A_T, bool B_T>
__device__ __forceinline__ void product64(const __half *At, const __half *Bt, int m0, int n0, float (&acc)[4][4])
{
    const int lane = threadIdx.x & 31, l8 = lane & 7, b3 = (lane >> 3) & 1, b4 = lane >> 4;
    const uint32_t a0 = (uint32_t)__cvta_generic_to_shared(At) + 2 * (A_T ? (l8 + 8 * b4) * LDH + m0 + 8 * b3 : (m0 + l8 + 8 * b3) * LDH + 8 * b4);
    const uint32_t b0 = (uint32_t)__cvta_generic_to_shared(Bt) + 2 * (B_T ? (n0 + l8 + 8 * b4) * LDH + 8 * b3 : (l8 + 8 * b3) * LDH + n0 + 8 * b4);
    constexpr uint32_t AS = 2 * (A_T ? 16 * LDH : 16), BS = 2 * (B_T ? 16 : 16 * LDH), BN = 2 * (B_T ? 16 * LDH : 16);
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) {
        uint32_t ah[4], al[4], bh[2][4], bl[2][4];
        ldsm4<A_T>(a0 + ks * AS, ah);
        ldsm4<A_T>(a0 + ks * AS + 2 * PLANE, al);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            ldsm4<!B_T>(b0 + ks * BS + j * BN, bh[j]);
            ldsm4<!B_T>(b0 + ks * BS + j * BN + 2 * PLANE, bl[j]);
        }
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) mma_f16(acc[nt], al, bh[nt >> 1][2 * (nt & 1)], bh[nt >> 1][2 * (nt & 1) + 1]);
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) mma_f16(acc[nt], ah, bl[nt >> 1][2 * (nt & 1)], bl[nt >> 1][2 * (nt & 1) + 1]);
#pragma unroll
        for (int nt = 0; nt < 4; ++nt) mma_f16(acc[nt], ah, bh[nt >> 1][2 * (nt & 1)], bh[nt >> 1][2 * (nt & 1) + 1]);
    }
}

// The same for a 16 x 16 part of the result and A = At.
template <bool B_T>
__device__ __forceinline__ void product16(const __half *At, const __half *Bt, int m0, int n0, float (&acc)[2][4])
{
    const int lane = threadIdx.x & 31, l8 = lane & 7, b3 = (lane >> 3) & 1, b4 = lane >> 4;
    const uint32_t a0 = (uint32_t)__cvta_generic_to_shared(At) + 2 * ((m0 + l8 + 8 * b3) * LDH + 8 * b4);
    const uint32_t b0 = (uint32_t)__cvta_generic_to_shared(Bt) + 2 * (B_T ? (n0 + l8 + 8 * b4) * LDH + 8 * b3 : (l8 + 8 * b3) * LDH + n0 + 8 * b4);
    constexpr uint32_t BS = 2 * (B_T ? 16 : 16 * LDH);
#pragma unroll
    for (int ks = 0; ks < 4; ++ks) {
        uint32_t ah[4], al[4], bh[4], bl[4];
        ldsm4<false>(a0 + ks * 32, ah);
        ldsm4<false>(a0 + ks * 32 + 2 * PLANE, al);
        ldsm4<!B_T>(b0 + ks * BS, bh);
        ldsm4<!B_T>(b0 + ks * BS + 2 * PLANE, bl);
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) mma_f16(acc[nt], al, bh[2 * nt], bh[2 * nt + 1]);
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) mma_f16(acc[nt], ah, bl[2 * nt], bl[2 * nt + 1]);
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) mma_f16(acc[nt], ah, bh[2 * nt], bh[2 * nt + 1]);
    }
}

// Power of two s with |x| s < 2^top for every |x| <= max (max given by its bits), and its inverse.
__device__ __forceinline__ float2 scale_for(unsigned max_bits, int top)
{
    const int e = (int)((max_bits >> 23) & 255u);                // max < 2^(e - 126)
    const int k = min(max(top + 126 - e, -120), 120);
    return make_float2(__int_as_float((127 + k) << 23), __int_as_float((127 - k) << 23));
}

}  // namespace hs
