// Warp-level fp32 matrix products on the tensor cores: every fp32 operand is split into two tf32
// parts (x = hi + lo, both rounded to nearest: 22 significant bits together) and a product takes three
// mma.sync m16n8k8 (hi hi + hi lo + lo hi) with fp32 accumulation.  The dropped lo lo term and the
// residue of the split are below 2^-22 of a product, i.e. of the size of fp32 rounding.
//
// Why mma.sync here: operands are plain fp32 arrays in shared memory that each product reads in
// another orientation, and a fragment is split in the registers it is loaded into, so no operand
// image is ever materialised.  Measured on B200: 490 tf32 MAC per clock and SM, 163 after the
// factor three, against 128 for FMA instructions that also have to share the issue slots with their
// operand loads.
#pragma once
#include <stdint.h>

namespace kda {
namespace mma3 {

__device__ __forceinline__ uint32_t tf32_rn(float x) {
    uint32_t r;
    asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ void split(float x, uint32_t& hi, uint32_t& lo) {
    hi = tf32_rn(x);
    lo = tf32_rn(x - __uint_as_float(hi));
}
__device__ __forceinline__ void mma8(float (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
    asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// acc[:, NO .. NO+NU) += A (16 MT rows) * B (8 NU columns) over k in [k0, k1) (multiples of 8).
// A(m, k) is A[m * lda + k], or A[k * lda + m] when AT; B(k, n) is B[k * ldb + n], or B[n * ldb + k]
// when BT.  AX / BX: every element of the operand is a tf32 number (bf16 data), its low part is zero
// and is skipped.  Free of bank conflicts for ld = 4 (mod 32) where k is the contiguous index and
// ld = 8 (mod 32) where it is not.
// Fragment layout: lane = 4 g + c; acc[mt][nt] = rows 16 mt + g (+8), columns 8 nt + 2 c (+1).
template <int NO, int NU, bool AT, bool BT, bool AX, bool BX, int MT, int NT>
__device__ __forceinline__ void gemm(float (&acc)[MT][NT][4], const float* __restrict__ A, int lda,
                                     const float* __restrict__ B, int ldb, int k0, int k1, int lane)
{
    const int g = lane >> 2, c = lane & 3;
    const int sam = AT ? 1 : lda, sak = AT ? lda : 1;
    const int sbn = BT ? ldb : 1, sbk = BT ? 1 : ldb;
    const float* pa = A + g * sam + (k0 + c) * sak;
    const float* pb = B + g * sbn + (k0 + c) * sbk;
#pragma unroll 2
    for (int k = k0; k < k1; k += 8, pa += 8 * sak, pb += 8 * sbk) {
        uint32_t ah[MT][4], al[MT][4], bh[NU][2], bl[NU][2];
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int j = 0; j < 4; ++j) {
                const float x = pa[(16 * m + 8 * (j & 1)) * sam + 4 * (j >> 1) * sak];
                if (AX) ah[m][j] = __float_as_uint(x);
                else split(x, ah[m][j], al[m][j]);
            }
#pragma unroll
        for (int n = 0; n < NU; ++n)
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const float x = pb[8 * n * sbn + 4 * j * sbk];
                if (BX) bh[n][j] = __float_as_uint(x);
                else split(x, bh[n][j], bl[n][j]);
            }
        // the tensor core truncates when it adds to its accumulator, so a step's products are summed from
        // zero, smallest first, and added to acc with rounding to nearest
        float tmp[MT][NU][4];
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int n = 0; n < NU; ++n) {
#pragma unroll
                for (int j = 0; j < 4; ++j) tmp[m][n][j] = 0.f;
                if (!BX) mma8(tmp[m][n], ah[m], bl[n]);
            }
        if (!AX)
#pragma unroll
            for (int m = 0; m < MT; ++m)
#pragma unroll
                for (int n = 0; n < NU; ++n) mma8(tmp[m][n], al[m], bh[n]);
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int n = 0; n < NU; ++n) {
                mma8(tmp[m][n], ah[m], bh[n]);
            }
#pragma unroll
        for (int m = 0; m < MT; ++m)
#pragma unroll
            for (int n = 0; n < NU; ++n)
#pragma unroll
                for (int j = 0; j < 4; ++j) acc[m][NO + n][j] += tmp[m][n][j];
    }
}

template <int MT, int NT>
__device__ __forceinline__ void zero(float (&acc)[MT][NT][4]) {
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[m][n][j] = 0.f;
}

}  // namespace mma3
}  // namespace kda
