// What the two translation units of the backward pass share: the arguments and the per-(chunk, head)
// scratch tile of the chunkwise form (kda_bwd_chunk.cu); kda_bwd.cu holds the entry point and the
// token-sequential form.
#pragma once
#include "kda_common.cuh"

namespace kda {

struct BwdChunkArgs {
    const void* q; const void* k; const void* v; const void* d_o;    // d_o may be nullptr (zeros)
    const float* log_alpha; const float* beta;
    const float* S0; const float* dS_T;                              // or nullptr (zeros)
    float* dq; float* dk; float* dv; float* dg; float* db; float* dS0;   // dS0 may be nullptr
    const int32_t* cu_seqlens; const int32_t* chunk_cu;              // nullptr = equal lengths
    float* tiles;                                                    // [chunks][H][kBwdTile]
    int* seq_heads;   // [H]: 1 = a chunk of this head decays too fast for the chunkwise form
    int n_seqs, H;
    WsHeader* hdr;
    int64_t seq_len, chunks_per_seq, n_chunks;
    float scale;
    unsigned long long wait_limit_ns;
};

// Scratch tile (floats), written by the first kernel unless stated otherwise
namespace bt {
constexpr int W = 0;                 // [64][128] W' = T' K^      (K^ = k e^G, T' = (I + StrictTril(K^ K~^T) Diag(beta))^-1)
constexpr int R = W + 64 * 128;      // [64][128] U' = T' V, replaced by r = U' - W' S by the forward chain
constexpr int X = R + 64 * 128;      // [64][128] Tril(Q K^T)^T dO, replaced by dX = .. + K~ Lam by the backward chain
constexpr int KT = X + 64 * 128;     // [64][128] K~ = k e^(G_C - G)
constexpr int N = KT + 64 * 128;     // [128][128] Q^T dO
constexpr int S = N + 128 * 128;     // [128][128] state entering the chunk (forward chain)
constexpr int L = S + 128 * 128;     // [128][128] adjoint of the state leaving the chunk (backward chain)
constexpr int G = L + 128 * 128;     // [64][128] cumulative log decay
constexpr int T = G + 64 * 128;      // [64][64] T'
constexpr int B = T + 64 * 64;       // [64][64] StrictTril(K^ K~^T)
constexpr int GC = B + 64 * 64;      // [128] e^(G_C)
constexpr int kFloats = GC + 128;
}  // namespace bt

// first token, valid tokens (1..64) and sequence of global chunk g
struct BwdLoc { int64_t tok0; int len; int n; };
__device__ __forceinline__ BwdLoc bwd_locate(const BwdChunkArgs& a, int64_t g) {
    BwdLoc L;
    int64_t c;
    int64_t b, e;
    if (a.cu_seqlens == nullptr) {
        L.n = (int)(g / a.chunks_per_seq);
        c = g - (int64_t)L.n * a.chunks_per_seq;
        b = (int64_t)L.n * a.seq_len; e = b + a.seq_len;
    } else {
        int lo = 0, hi = a.n_seqs - 1;   // last n with chunk_cu[n] <= g
        while (lo < hi) {
            const int mid = (lo + hi + 1) >> 1;
            if ((int64_t)a.chunk_cu[mid] <= g) lo = mid; else hi = mid - 1;
        }
        L.n = lo;
        c = g - a.chunk_cu[lo];
        b = a.cu_seqlens[lo]; e = a.cu_seqlens[lo + 1];
    }
    L.tok0 = b + c * kC;
    L.len = (e - L.tok0) < kC ? (int)(e - L.tok0) : kC;

    return L;
}

kda_status_t launch_bwd_out(const BwdChunkArgs& a, kda_dtype_t dt, cudaStream_t st);
kda_status_t launch_bwd_chunk(const BwdChunkArgs& a, kda_dtype_t dt, int32_t* chunk_cu_dev, cudaStream_t st);

}  // namespace kda
