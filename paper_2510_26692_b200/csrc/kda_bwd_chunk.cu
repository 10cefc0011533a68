// Chunkwise backward pass (adjoint of the chunk form of paper Section 3.1; the paper prints no
// backward algorithm).  Notation of one 64-token chunk of one head, G the cumulative log decay:
//     K^ = k e^G, K_ = k e^-G, K~ = k e^(G_C - G), Q = scale q e^G,  B = StrictTril(K^ K_^T), P = Tril(Q K_^T)
//     r  = T' (V - K^ S),  T' = (I + B Diag(beta))^-1       residuals v_t - S'_t^T k_t of Eq. 1
//     S+ = e^(G_C) S + K~^T (beta r),   O = Q S + P (beta r)
// With Lam the adjoint of S+ and dO that of O:
//     dX  = P^T dO + K~ Lam             dV  = T'^T (beta dX)
//     Lam-= e^(G_C) Lam + Q^T dO - W'^T (beta dX),  W' = T' K^   (the adjoint of S: same form as S+)
//     dP  = Tril(dO (beta r)^T)         dB  = -StrictTril(dV (beta r)^T)
//     dQ  = dO S^T + dP K_              dK^ = -dV S^T + dB K_
//     dK_ = dP^T Q + dB^T K^            dK~ = (beta r) Lam^T
//     dbeta_j = r_j . dX_j - sum_i B_ij (dV_i . r_j)
//     dG_i = q dq + k (the K^ share of dk - the K_ and K~ shares);  dG_C adds sum_i K~ dK~ + e^(G_C) rowsum(S Lam)
//     dlog_alpha_i = sum_{j >= i} dG_j
// Three kernels: what is local to a chunk (kda_bwd_intra.cu, all chunks at once), the two state recurrences
// (kda_bwd_chain.cu, forward and backward chains side by side) and the gradients (kda_bwd_out.cu, all chunks
// at once).  e^G and e^-G are taken relative to the middle of the chunk's decay range.  A head with a chunk
// whose log decay leaves [-kBwdRange, 1], or with a token that is not finite, is left to the token-sequential kernels
// (kda_bwd.cu).
#include "kda_bwd.cuh"
#include "kda_ptx.cuh"

namespace kda {
namespace {

// clears the status word and the per-head marks, builds the chunk table of a packed batch
__global__ void kda_bwd_prep(WsHeader* hdr, const int32_t* cu, int32_t* chunk_cu, int n_seqs,
                             int* seq_heads, int H)
{
    ptx::grid_dep_wait();      // (launched before the preceding kernel has ended)
    ptx::grid_dep_launch();
    for (int h = threadIdx.x; h < H; h += blockDim.x) seq_heads[h] = 0;
    if (threadIdx.x == 0) {
        hdr->status = 0; hdr->where = 0; hdr->flags = 0;
        if (cu) {
            int acc = 0;
            chunk_cu[0] = 0;
            for (int n = 0; n < n_seqs; ++n) {
                acc += (cu[n + 1] - cu[n] + kC - 1) / kC;
                chunk_cu[n + 1] = acc;
            }
        }
    }
}

}  // namespace

kda_status_t launch_bwd_chunk(BwdChunkArgs a, kda_dtype_t dt, int32_t* chunk_cu_dev, cudaStream_t st)
{
    {
        DeviceLock lk;
        if (!lk.st) return lk.rc;
        if (lk.st->n_sm == 0) {
            int dev = 0;
            KDA_CUDA_TRY(cudaGetDevice(&dev));
            KDA_CUDA_TRY(cudaDeviceGetAttribute(&lk.st->n_sm, cudaDevAttrMultiProcessorCount, dev));
        }
        a.n_sm = lk.st->n_sm;
    }
    KDA_CUDA_TRY(launch_dependent(kda_bwd_prep, dim3(1), 256, 0, st, a.hdr, a.cu_seqlens, chunk_cu_dev, a.n_seqs, a.seq_heads, a.H));
    count_launch();
    kda_status_t rc = a.n_chunks > 0 ? launch_bwd_intra(a, dt, st) : KDA_OK;
    if (rc == KDA_OK) rc = launch_bwd_chain(a, st);
    if (rc == KDA_OK && a.n_chunks > 0) rc = launch_bwd_out(a, dt, st);
    return rc;
}

}  // namespace kda
