// Layout of the per-(chunk, head) scratch tile that the intra-chunk stage hands to the inter-chunk
// stage on the bf16 tensor-core path.  Every matrix operand is stored as the exact shared-memory
// image the tcgen05 MMA expects (128-byte swizzle, see ptx::sw128_off), so the consumer brings the whole tile
// in with one 1-D bulk copy.
#pragma once
#include <stdint.h>

namespace kda {
namespace tc {
// [ W ; Q ] = [ T Diag(beta) (Gamma.K) ; scale Gamma.Q ]: two K-halves of [128 rows][64], rows 0-63 = W, 64-127 = Q
constexpr uint32_t OFF_QW = 0;
constexpr uint32_t QW_HALF = 128 * 128;
// layer calls of few chains: the chunk's output rows in fp32, over [ W ; Q ] once the chain has read them; element
// (token, column) at float ((token / 4) 128 + column) 4 + token % 4
constexpr uint32_t OFF_O32 = OFF_QW;
// K' = K exp(G_m - G), relative to the middle G_m of the chunk's log-decay range (the reference of the decay
// factorisation: G_C / 2 as a whole number of halvings), as two dk-halves of [64 tokens][64 channels]; the consumer restores exp(G_C - G_m) in fp32
constexpr uint32_t OFF_KI = 32768;
constexpr uint32_t KI_HALF = 64 * 128;
// Aqk [64][64] (lower triangular incl. diagonal)
constexpr uint32_t OFF_AQ = 49152;
// gamma^C = exp(G_C) and exp(G_C - G_m), 128 fp32 each
constexpr uint32_t OFF_GV = 57344;
constexpr uint32_t GV_BYTES = 1024;
// U^T: 16-byte chunk c holds tokens 8 c .. 8 c + 7 of column `col`; read with plain loads, a thread per column
constexpr uint32_t OFF_U = OFF_GV + GV_BYTES;
__host__ __device__ __forceinline__ constexpr uint32_t ut_off(uint32_t col, uint32_t chunk) { return (chunk * 128u + col) << 4; }
constexpr uint32_t TILE_BYTES = OFF_U + 16384;
static_assert(TILE_BYTES % 256 == 0, "tiles stay 256-byte aligned");
}  // namespace tc
}  // namespace kda
