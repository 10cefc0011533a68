// fp32 matrix products on tcgen05: every fp32 operand is stored as three bf16 images in shared memory,
// x = x1 + x2 + x3 with each part rounded to nearest (24 significant bits together), and a product takes
// the six MMAs x1 y1, x1 y2, x2 y1, x2 y2, x1 y3, x3 y1 into one fp32 accumulator in TMEM, small ones
// first, so that the accumulator is truncated at full size by the last group alone (by all six where a product is added
// to one that is complete).  The dropped terms are below 2^-25 of a product.
//
// An image is a sequence of blocks [R rows][64 columns] bf16 with 128-byte rows and the 128-byte swizzle;
// split s, column block b of a matrix with NB column blocks start at (s * NB + b) * R * 128 bytes.  The
// same image serves as K-major operand (rows = M or N, columns = K) and as MN-major operand
// (rows = K, columns = M or N).
//
// Six bf16 MMAs per product leave 1/6 of the bf16 rate, 680 MAC per clock and SM, against 163 for three
// warp-level tf32 MMAs (kda_mma3.cuh), and an operand is split once instead of by every warp that reads it.
#pragma once
#include <cuda_bf16.h>

#include "kda_ptx.cuh"

namespace kda {
namespace split3 {

__device__ __forceinline__ uint32_t pack2(float lo, float hi) {
    uint32_t r;
    asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
    return r;
}
// The next split of a pair of values: returns it and leaves the rest in r (one packed operation).
__device__ __forceinline__ uint32_t take2(float2& r) {
    const uint32_t w = pack2(r.x, r.y);
    r = __ffma2_rn(make_float2(__uint_as_float(w << 16), __uint_as_float(w & 0xffff0000u)), make_float2(-1.f, -1.f), r);
    return w;
}
// Splits x[0..7] into the 16-byte chunk (row, col .. col+7) of a matrix image, col a multiple of 8.
template <int R, int NB>
__device__ __forceinline__ void put8(uint8_t* img, int row, int col, const float (&x)[8]) {
    uint8_t* p = img + (col >> 6) * (R * 128) + ptx::sw128_off((uint32_t)row, (uint32_t)(col & 63));
    float2 r[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) r[e] = make_float2(x[2 * e], x[2 * e + 1]);
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        uint32_t w[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) w[e] = s < 2 ? take2(r[e]) : pack2(r[e].x, r[e].y);
        *reinterpret_cast<uint4*>(p + s * (NB * R * 128)) = make_uint4(w[0], w[1], w[2], w[3]);
    }
}
// Splits 16 or 32 consecutive columns of this lane's row into the A operand in TMEM (two bf16 values a column, kParts columns
// from one split to the next): no pass over shared memory, and the product reads only its B operand there.
// `written(s)` is called behind the store of split s.
template <int kParts, int N, typename F>
__device__ __forceinline__ void put_tmem(uint32_t taddr, const float2 (&x)[N], F written) {
    static_assert(N == 8 || N == 16, "a tcgen05.st of 8 or 16 columns");
    float2 r[N];
#pragma unroll
    for (int e = 0; e < N; ++e) r[e] = x[e];
#pragma unroll
    for (int s = 0; s < 3; ++s) {
        uint32_t w[N];
#pragma unroll
        for (int e = 0; e < N; ++e) w[e] = s < 2 ? take2(r[e]) : pack2(r[e].x, r[e].y);
        if constexpr (N == 16) ptx::tmem_st_32x32b_x16(taddr + s * kParts, w);
        else ptx::tmem_st_32x32b_x8(taddr + s * kParts, w);
        written(s);
    }
}
template <int kParts, int N>
__device__ __forceinline__ void put_tmem(uint32_t taddr, const float2 (&x)[N]) {
    put_tmem<kParts>(taddr, x, [](int) {});
}

// One operand of a product: descriptor of split 0 at K = 0, and the distances between splits and of 16 in K
// (in descriptor units of 16 bytes).  KH: distance of the second 64 of K (K-major operands).
struct Operand {
    uint64_t desc;
    uint32_t split, k16, khalf;
};
template <int R, int NB>
__device__ __forceinline__ Operand k_major(const uint8_t* img, int row0 = 0) {
    return {ptx::umma_desc_sw128(ptx::smem_u32(img) + row0 * 128), NB * R * 8u, 2u, R * 8u};
}
// `dup`: both 64-blocks of M read column block 0 (TMEM lanes 64-127 then repeat lanes 0-63)
template <int R, int NB>
__device__ __forceinline__ Operand mn_major(const uint8_t* img, int row0 = 0, bool dup = false) {
    return {ptx::umma_desc_sw128_mn(ptx::smem_u32(img) + row0 * 128, dup ? 0u : R * 128u), NB * R * 8u, 128u, 512u};
}

// d (+)= A B over KS steps of 16 in K; a whole converged warp.  idesc carries M, N and the majors.  kExactA: A holds bf16
// numbers, its image the first split alone (three MMAs).
template <int KS, bool kExactA = false>
__device__ __forceinline__ void mma6(uint32_t d_tmem, const Operand& A, const Operand& B, uint32_t idesc, bool accumulate) {
    // (sa, sb): (2,0) (0,2) (1,1) (1,0) (0,1) (0,0); exact: (0,2) (0,1) (0,0)
    uint32_t acc = accumulate ? 1u : 0u;
#pragma unroll 1
    for (int p = 0; p < (kExactA ? 3 : 6); ++p) {
        const uint32_t sa = kExactA ? 0u : p == 0 ? 2u : (p == 2 || p == 3) ? 1u : 0u;
        const uint32_t sb = kExactA ? 2u - p : p == 1 ? 2u : (p == 2 || p == 4) ? 1u : 0u;
        const uint64_t da = A.desc + sa * A.split, db = B.desc + sb * B.split;
#pragma unroll
        for (int k = 0; k < KS; ++k) {
            const uint32_t oa = A.k16 == 2u ? (uint32_t)(k >> 2) * A.khalf + (k & 3) * 2u : (uint32_t)k * A.k16;
            const uint32_t ob = B.k16 == 2u ? (uint32_t)(k >> 2) * B.khalf + (k & 3) * 2u : (uint32_t)k * B.k16;
            ptx::umma_bf16(d_tmem, da + oa, db + ob, idesc, acc);
            acc = 1u;
        }
    }
}

// one of the six with A in TMEM (put_tmem): split sa of A, split sb of B
template <int KS, int kParts>
__device__ __forceinline__ void mma_ta(uint32_t d_tmem, uint32_t a_tmem, const Operand& B, uint32_t idesc, uint32_t sa, uint32_t sb, bool accumulate) {
    uint32_t acc = accumulate ? 1u : 0u;
    const uint32_t ta = a_tmem + sa * kParts;
    const uint64_t db = B.desc + sb * B.split;
#pragma unroll
    for (int k = 0; k < KS; ++k) {
        const uint32_t ob = B.k16 == 2u ? (uint32_t)(k >> 2) * B.khalf + (k & 3) * 2u : (uint32_t)k * B.k16;
        ptx::umma_bf16_ta(d_tmem, ta + k * 8, db + ob, idesc, acc);
        acc = 1u;
    }
}
// all six, those with the splits of A that are written first at the start: (0,2) (1,1) (2,0) (1,0) (0,1) (0,0); `ready(s)`
// comes before the first that needs split s
template <int KS, int kParts, typename F>
__device__ __forceinline__ void mma6_ta(uint32_t d_tmem, uint32_t a_tmem, const Operand& B, uint32_t idesc, bool accumulate, F ready) {
#pragma unroll 1
    for (int p = 0; p < 6; ++p) {
        if (p < 3) ready(p);
        const uint32_t sa = p < 3 ? p : p == 3 ? 1u : 0u, sb = p < 3 ? 2u - p : p == 4 ? 1u : 0u;
        mma_ta<KS, kParts>(d_tmem, a_tmem, B, idesc, sa, sb, accumulate || p > 0);
    }
}
template <int KS, int kParts>
__device__ __forceinline__ void mma6_ta(uint32_t d_tmem, uint32_t a_tmem, const Operand& B, uint32_t idesc, bool accumulate) {
    mma6_ta<KS, kParts>(d_tmem, a_tmem, B, idesc, accumulate, [](int) {});
}

}  // namespace split3
}  // namespace kda
