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

// The high part is rounded to nearest (ties away) by an integer addition on the bit pattern; the tensor core ignores
// the 13 low bits.  (cvt.rna.tf32 gives the same and is several times slower to issue.)  The same addition would make
// minus zero of a NaN as the GPU's arithmetic writes it (0x7fffffff), and the product would be finite.  So the low
// part, a NaN for every x that is not finite, is rounded by a multiplication: with 1 + 0.7 2^-11 before the cut its
// error is 0.31 of a step (root mean square; rounding to nearest: 0.29).
__device__ __forceinline__ void split(float x, uint32_t& hi, uint32_t& lo) {
    hi = (__float_as_uint(x) + 0x1000u) & 0xffffe000u;
    lo = __float_as_uint((x - __uint_as_float(hi)) * 1.00034180f);
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
    // (steps depend on each other through the additions to acc alone: small blocks overlap more of them)
    constexpr int kUnroll = MT * NU == 1 ? 4 : 2;
#pragma unroll kUnroll
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

// f(row, column, x, y) for every pair of neighbouring columns that this lane holds of a fragment block
template <int MT, int NT, typename F>
__device__ __forceinline__ void each_pair(const float (&acc)[MT][NT][4], int lane, F f) {
    const int g = lane >> 2, c = lane & 3;
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            f(16 * m + g, 8 * n + 2 * c, acc[m][n][0], acc[m][n][1]);
            f(16 * m + g + 8, 8 * n + 2 * c, acc[m][n][2], acc[m][n][3]);
        }
}
__device__ __forceinline__ void st2(float* p, float x, float y) { *reinterpret_cast<float2*>(p) = make_float2(x, y); }

// T = (I + L)^-1 of a strictly lower triangular 64 x 64 L (row pitch LD, its upper triangle is overwritten), by
// at least 4 warps; T has to be zero above the diagonal blocks on entry.  16 x 16 diagonal blocks by substitution
// (one column per thread, fp32 FMA), then two doublings [T11 0; T21 T22], T21 = -T22 (L21 T11), as warp-level
// products whose inner factor sits in the empty upper triangle of L.  `barrier` is one of all calling threads; ends with it.  (With the
// doublings as FMA products over all threads: 11.1k cycles instead of 8.0k.)
template <int LD, typename Barrier>
__device__ __forceinline__ void invert_unit_lower(float* __restrict__ L, float* __restrict__ T, int t, Barrier barrier) {
    const int lane = t & 31, w = t >> 5;
    if (t < 64) {
        const int b0 = t & 48, j = t & 15;
        float x[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            float s0 = i == j ? 1.f : 0.f, s1 = 0.f;
#pragma unroll
            for (int m = 0; m < i; ++m) {
                const float l = L[(b0 + i) * LD + b0 + m];
                if (m & 1) s1 = fmaf(-l, x[m], s1); else s0 = fmaf(-l, x[m], s0);
            }
            x[i] = s0 + s1;
        }
#pragma unroll
        for (int i = 0; i < 16; ++i) T[(b0 + i) * LD + b0 + j] = x[i];
    }
    barrier();
#pragma unroll
    for (int s = 16; s < 64; s *= 2) {
        // 16 x 16 block (i0, j0) of the pair at c0: two warps for s = 16, four for s = 32
        const int c0 = s == 16 ? 32 * w : 0, i0 = s == 16 ? 0 : 16 * (w >> 1), j0 = s == 16 ? 0 : 16 * (w & 1);
        const bool mine = w < (s == 16 ? 2 : 4);
        float acc[1][2][4];
        if (mine) {
            zero(acc);
            gemm<0, 2, false, false, false, false>(acc, L + (c0 + s + i0) * LD + c0, LD, T + c0 * LD + c0 + j0, LD, j0, s, lane);
            each_pair(acc, lane, [&](int i, int j, float x, float y) { st2(L + (c0 + i0 + i) * LD + c0 + s + j0 + j, x, y); });
        }
        barrier();
        if (mine) {
            zero(acc);
            gemm<0, 2, false, false, false, false>(acc, T + (c0 + s + i0) * LD + c0 + s, LD, L + c0 * LD + c0 + s + j0, LD, 0,
                                                   i0 + 16, lane);
            each_pair(acc, lane, [&](int i, int j, float x, float y) { st2(T + (c0 + s + i0 + i) * LD + c0 + j0 + j, -x, -y); });
        }
        barrier();
    }
}

__device__ __forceinline__ void cp16(float* dst, const float* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
__device__ __forceinline__ void cp_wait0() { asm volatile("cp.async.wait_group 0;" ::: "memory"); }

}  // namespace mma3
}  // namespace kda
