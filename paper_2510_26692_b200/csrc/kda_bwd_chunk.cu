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
// Three kernels: what is local to a chunk (all chunks at once), the two state recurrences (forward
// and backward chains side by side, one CTA per column slice), and the gradients (all chunks at once).
// e^G and e^-G are taken relative to the middle of the chunk's decay range.  A head with a chunk whose
// log decay leaves [-kRange, 1] is left to the token-sequential kernels.  Products: kda_mma3.cuh.
#include "kda_bwd.cuh"
#include "kda_mma3.cuh"

namespace kda {
namespace {

using namespace mma3;

// Largest decay of a chunk taken in chunk form.  The cumulative sum is rounded to 2^-24 of its size, so
// every decay ratio carries a relative error of up to kRange 2^-24 = 2.4e-6.
constexpr float kRange = 40.f;

template <typename T> __device__ __forceinline__ float ldf(const T* p);
template <> __device__ __forceinline__ float ldf<float>(const float* p) { return *p; }
template <> __device__ __forceinline__ float ldf<__nv_bfloat16>(const __nv_bfloat16* p) { return __bfloat162float(*p); }

// clears the status word and the per-head marks, builds the chunk table of a packed batch
__global__ void kda_bwd_prep(WsHeader* hdr, const int32_t* __restrict__ cu, int32_t* __restrict__ chunk_cu, int n_seqs,
                             int* __restrict__ seq_heads, int H)
{
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

// ---- per-chunk stage -------------------------------------------------------------------------------
constexpr int kT1 = 512;
constexpr int LR = 132, LC = 136, LM = 68;       // row pitches: k-contiguous, k-strided, 64 x 64
namespace p1 {
constexpr int KG = 0;                            // K^ relative to the middle of the decay range  [64][LR]
constexpr int KI = KG + 64 * LR;                 // K_                                             [64][LR]
constexpr int QG = KI + 64 * LR;                 // Q                                              [64][LR]
constexpr int V = QG + 64 * LR;                  // [64][LC]
constexpr int DO = V + 64 * LC;                  // [64][LC]
constexpr int B = DO + 64 * LC;                  // [64][LM] B, later B Diag(beta)
constexpr int P = B + 64 * LM;                   // [64][LM]
constexpr int T = P + 64 * LM;                   // [64][LM] T'
constexpr int VEC = T + 64 * LM;                 // e^(G_m) [128], beta [64], segment sums [4][128]
constexpr int kFloats = VEC + 128 + 64 + 512;
}  // namespace p1
constexpr size_t kSmem1 = (size_t)p1::kFloats * 4;
static_assert(kSmem1 <= 232448, "fits the shared memory of one SM");

template <typename T>
__global__ void __launch_bounds__(kT1, 1) kda_bwd_intra(BwdChunkArgs a)
{
    constexpr bool kX = sizeof(T) == 2;          // stored bf16: v and d_o are tf32 numbers
    extern __shared__ __align__(16) float sm[];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const int h = blockIdx.y;
    const BwdLoc loc = bwd_locate(a, blockIdx.x);
    float* tile = a.tiles + ((size_t)blockIdx.x * a.H + h) * bt::kFloats;
    float* sKG = sm + p1::KG; float* sKI = sm + p1::KI; float* sQG = sm + p1::QG;
    float* sV = sm + p1::V; float* sDO = sm + p1::DO;
    float* sB = sm + p1::B; float* sP = sm + p1::P; float* sT = sm + p1::T;
    float* sEm = sm + p1::VEC; float* sBeta = sEm + 128; float* sSeg = sBeta + 64;

    // gates, k, q: thread = channel c of 16 consecutive tokens
    {
        const int c = t & 127, seg = t >> 7;
        const T* kp = reinterpret_cast<const T*>(a.k);
        const T* qp = reinterpret_cast<const T*>(a.q);
        float G[16], kk[16], qq[16];
        float run = 0.f, lo = 0.f, hi = 0.f;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const int r = seg * 16 + i;
            const size_t off = ((size_t)(loc.tok0 + r) * a.H + h) * kD + c;
            const bool in = r < loc.len;
            G[i] = in ? a.log_alpha[off] : 0.f;
            kk[i] = in ? ldf<T>(kp + off) : 0.f;
            qq[i] = in ? ldf<T>(qp + off) : 0.f;
        }
        // v and d_o: 16 float4 columns per row of 32 lanes
        for (int idx = t; idx < 64 * 32; idx += kT1) {
            const int r = idx >> 5, c4 = (idx & 31) * 4;
            float4 x = make_float4(0.f, 0.f, 0.f, 0.f), y = x;
            if (r < loc.len) {
                const size_t off = ((size_t)(loc.tok0 + r) * a.H + h) * kD + c4;
                x = IO<T>::load4(reinterpret_cast<const T*>(a.v) + off);
                if (a.d_o) y = IO<T>::load4(reinterpret_cast<const T*>(a.d_o) + off);
            }
            *reinterpret_cast<float4*>(sV + r * LC + c4) = x;
            *reinterpret_cast<float4*>(sDO + r * LC + c4) = y;
        }
        if (t < 64) sBeta[t] = t < loc.len ? a.beta[(size_t)(loc.tok0 + t) * a.H + h] : 0.f;
#pragma unroll
        for (int i = 0; i < 16; ++i) { run += G[i]; G[i] = run; }
        sSeg[seg * 128 + c] = run;
        __syncthreads();
        float base = 0.f, total = 0.f;
#pragma unroll
        for (int s = 0; s < 4; ++s) {
            const float x = sSeg[s * 128 + c];
            if (s < seg) base += x;
            total += x;
        }
        const float gm = 0.5f * total;
        const float em = expf(gm);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const int r = seg * 16 + i;
            G[i] += base;
            lo = fminf(lo, G[i]); hi = fmaxf(hi, G[i]);
            tile[bt::G + r * kD + c] = G[i];
            const float e1 = expf(G[i] - gm), e2 = expf(gm - G[i]);
            sKG[r * LR + c] = kk[i] * e1;
            sKI[r * LR + c] = kk[i] * e2;
            sQG[r * LR + c] = a.scale * qq[i] * e1;
            tile[bt::KT + r * kD + c] = kk[i] * expf(total - G[i]);
        }
        if (!(lo >= -kRange && hi <= 1.f && total - total == 0.f)) a.seq_heads[h] = 1;
        if (seg == 0) {
            sEm[c] = em;
            tile[bt::GC + c] = expf(total);
        }
        for (int idx = t; idx < 64 * LM; idx += kT1) sT[idx] = 0.f;
    }
    __syncthreads();

    // Gram matrices [K^ ; Q] K_^T: warps 4 x 4, 32 x 16 entries each; only blocks that reach the triangle
    {
        const int mi = w >> 2, ni = w & 3;
        const int r0 = (mi & 1) * 32, c0 = ni * 16;
        float acc[2][2][4];
        zero(acc);
        if (c0 < r0 + 32)
            gemm<0, 2, false, true, false, false>(acc, (mi < 2 ? sKG : sQG) + r0 * LR, LR, sKI + c0 * LR, LR, 0, kD, lane);
        float* dst = mi < 2 ? sB : sP;
        const int strict = mi < 2 ? 1 : 0;
        each_pair(acc, lane, [&](int i, int j, float x, float y) {
            i += r0; j += c0;
            x = j + strict <= i ? x : 0.f;
            y = j + 1 + strict <= i ? y : 0.f;
            if (mi < 2) {
                st2(tile + bt::B + i * 64 + j, x, y);
                x *= sBeta[j]; y *= sBeta[j + 1];
            }
            st2(dst + i * LM + j, x, y);
        });
    }
    __syncthreads();

    invert_unit_lower<kT1, LM>(sB, sT, t);      // T' = (I + B Diag(beta))^-1
    for (int idx = t; idx < 64 * 64; idx += kT1) tile[bt::T + idx] = sT[(idx >> 6) * LM + (idx & 63)];

    // W' = T' K^, U' = T' V, P^T dO: warps 2 x 8, 32 x 16 entries each; the triangles bound the sums
    {
        const int r0 = (w >> 3) * 32, c0 = (w & 7) * 16;
        float acc[2][2][4];
        zero(acc);
        gemm<0, 2, false, false, false, false>(acc, sT + r0 * LM, LM, sKG + c0, LR, 0, r0 + 32, lane);
        each_pair(acc, lane, [&](int i, int j, float x, float y) {
            st2(tile + bt::W + (r0 + i) * kD + c0 + j, x * sEm[c0 + j], y * sEm[c0 + j + 1]);
        });
        zero(acc);
        gemm<0, 2, false, false, false, kX>(acc, sT + r0 * LM, LM, sV + c0, LC, 0, r0 + 32, lane);
        each_pair(acc, lane, [&](int i, int j, float x, float y) { st2(tile + bt::R + (r0 + i) * kD + c0 + j, x, y); });
        zero(acc);
        gemm<0, 2, true, false, false, kX>(acc, sP + r0, LM, sDO + c0, LC, r0, 64, lane);
        each_pair(acc, lane, [&](int i, int j, float x, float y) { st2(tile + bt::X + (r0 + i) * kD + c0 + j, x, y); });
    }
    // Q^T dO: warps 4 x 4, 32 x 32 entries each
    {
        const int r0 = (w >> 2) * 32, c0 = (w & 3) * 32;
        float acc[2][4][4];
        zero(acc);
        gemm<0, 4, true, false, false, kX>(acc, sQG + r0, LR, sDO + c0, LC, 0, 64, lane);
        each_pair(acc, lane, [&](int i, int j, float x, float y) {
            const float e = sEm[r0 + i];
            st2(tile + bt::N + (r0 + i) * kD + c0 + j, x * e, y * e);
        });
    }
}

// ---- the two chains -----------------------------------------------------------------------------------
// State columns never mix: CTA = (column slice, head, sequence, direction).  The state lives in the
// accumulator fragments of the second product (8 warps as 4 x 2), with a copy in shared memory as the B
// operand of the first.  The next chunk's operands arrive by cp.async meanwhile.
constexpr int kT2 = 256;
template <int NS> struct ChainSmem {
    static constexpr int LS = NS + 8;
    static constexpr int A1 = 0;                     // [64][LR] W' (forward) / K~ (backward)
    static constexpr int A2 = A1 + 64 * LR;          // [64][LC] K~ (forward) / W' (backward)
    static constexpr int Y = A2 + 64 * LC;           // [64][LS] U' or P^T dO, replaced by beta r or -beta dX
    static constexpr int kStage = Y + 64 * LS;
    static constexpr int ST = 2 * kStage;            // [128][LS] state
    static constexpr size_t kBytes = (size_t)(ST + 128 * LS) * 4;
};
static_assert(ChainSmem<64>::kBytes <= 232448, "fits the shared memory of one SM");

template <int NS, bool kFwd>
__device__ __forceinline__ void chain_run(const BwdChunkArgs& a, float* sm, int n, int h, int col0)
{
    using M = ChainSmem<NS>;
    constexpr int LS = M::LS, NT = NS / 16;
    const int t = threadIdx.x, lane = t & 31, w = t >> 5, mi = w >> 1, ni = w & 1;
    const int g = lane >> 2, c2 = 2 * (lane & 3);
    int64_t g0, nc, tok_begin, tok_end;
    if (a.cu_seqlens) {
        g0 = a.chunk_cu[n]; nc = a.chunk_cu[n + 1] - g0;
        tok_begin = a.cu_seqlens[n]; tok_end = a.cu_seqlens[n + 1];
    } else {
        g0 = (int64_t)n * a.chunks_per_seq; nc = a.chunks_per_seq;
        tok_begin = (int64_t)n * a.seq_len; tok_end = tok_begin + a.seq_len;
    }
    const size_t sbase = ((size_t)n * a.H + h) * (size_t)(kD * kD);
    const int row2 = 32 * mi, ncol = ni * (NS / 2);      // this warp's block of the state
    float* sS = sm + M::ST;
    auto tile_of = [&](int64_t c) { return a.tiles + ((size_t)(g0 + c) * a.H + h) * bt::kFloats; };
    auto fetch = [&](int64_t c, int stage) {
        const float* tile = tile_of(c);
        float* s = sm + stage * M::kStage;
        const float* p1 = tile + (kFwd ? bt::W : bt::KT);
        const float* p2 = tile + (kFwd ? bt::KT : bt::W);
        for (int idx = t; idx < 64 * 32; idx += kT2) {
            const int r = idx >> 5, x = (idx & 31) * 4;
            cp16(s + M::A1 + r * LR + x, p1 + r * kD + x);
            cp16(s + M::A2 + r * LC + x, p2 + r * kD + x);
        }
        const float* py = tile + (kFwd ? bt::R : bt::X) + col0;
        for (int idx = t; idx < 64 * (NS / 4); idx += kT2) {
            const int r = idx / (NS / 4), x = (idx % (NS / 4)) * 4;
            cp16(s + M::Y + r * LS + x, py + r * kD + x);
        }
        cp_commit();
    };

    float S[2][NT][4];
    const float* init = kFwd ? a.S0 : a.dS_T;
#pragma unroll
    for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
                const int r = row2 + 16 * m + 8 * hf + g, x = ncol + 8 * nt + c2;
                float2 v = make_float2(0.f, 0.f);
                if (init) v = *reinterpret_cast<const float2*>(init + sbase + (size_t)r * kD + col0 + x);
                S[m][nt][2 * hf] = v.x; S[m][nt][2 * hf + 1] = v.y;
                st2(sS + r * LS + x, v.x, v.y);
            }
    if (nc > 0) fetch(kFwd ? 0 : nc - 1, 0);
    for (int64_t i = 0; i < nc; ++i) {
        const int64_t c = kFwd ? i : nc - 1 - i;
        float* tile = tile_of(c);
        float* stage = sm + (i & 1) * M::kStage;
        cp_wait0();
        __syncthreads();      // this chunk's operands and the state are in place; the other stage is free
        if (i + 1 < nc) fetch(kFwd ? c + 1 : c - 1, (int)((i + 1) & 1));
        float gam[4], bt2[2];
        float2 nn[kFwd ? 1 : 2][kFwd ? 1 : NT][2];
#pragma unroll
        for (int j = 0; j < 4; ++j) gam[j] = tile[bt::GC + row2 + 8 * j + g];
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int64_t tok = tok_begin + c * kC + 16 * mi + 8 * j + g;
            bt2[j] = tok < tok_end ? a.beta[(size_t)tok * a.H + h] : 0.f;
        }
        if (!kFwd) {
#pragma unroll
            for (int m = 0; m < (kFwd ? 1 : 2); ++m)
#pragma unroll
                for (int nt = 0; nt < (kFwd ? 1 : NT); ++nt)
#pragma unroll
                    for (int hf = 0; hf < 2; ++hf)
                        nn[m][nt][hf] = *reinterpret_cast<const float2*>(
                            tile + bt::N + (row2 + 16 * m + 8 * hf + g) * kD + col0 + ncol + 8 * nt + c2);
        }
        float* keep = tile + (kFwd ? bt::S : bt::L) + col0;
        each_pair(S, lane, [&](int r, int x, float u, float v) { st2(keep + (row2 + r) * kD + ncol + x, u, v); });
        // first product: 64 rows, 16 per warp
        float y[1][NT][4];
        zero(y);
        gemm<0, NT, false, false, false, false>(y, stage + M::A1 + 16 * mi * LR, LR, sS + ncol, LS, 0, kD, lane);
        float* sY = stage + M::Y;
        float* out = tile + (kFwd ? bt::R : bt::X) + col0;
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
                const int r = 16 * mi + 8 * hf + g, x = ncol + 8 * nt + c2;
                float2 u = *reinterpret_cast<float2*>(sY + r * LS + x);
                if (kFwd) { u.x -= y[0][nt][2 * hf]; u.y -= y[0][nt][2 * hf + 1]; }
                else { u.x += y[0][nt][2 * hf]; u.y += y[0][nt][2 * hf + 1]; }
                *reinterpret_cast<float2*>(out + r * kD + x) = u;
                const float f = kFwd ? bt2[hf] : -bt2[hf];
                st2(sY + r * LS + x, f * u.x, f * u.y);
            }
        __syncthreads();
        // second product into the state
#pragma unroll
        for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int nt = 0; nt < NT; ++nt)
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) {
                    const float gg = gam[2 * m + hf];
                    float& s0 = S[m][nt][2 * hf];
                    float& s1 = S[m][nt][2 * hf + 1];
                    s0 *= gg; s1 *= gg;
                    if (!kFwd) { s0 += nn[kFwd ? 0 : m][kFwd ? 0 : nt][hf].x; s1 += nn[kFwd ? 0 : m][kFwd ? 0 : nt][hf].y; }
                }
        gemm<0, NT, true, false, false, false>(S, stage + M::A2 + row2, LC, sY + ncol, LS, 0, kC, lane);
        each_pair(S, lane, [&](int r, int x, float u, float v) { st2(sS + (row2 + r) * LS + ncol + x, u, v); });
    }
    if (!kFwd && a.dS0)
        each_pair(S, lane, [&](int r, int x, float u, float v) {
            st2(a.dS0 + sbase + (size_t)(row2 + r) * kD + col0 + ncol + x, u, v);
        });
}

template <int NS>
__global__ void __launch_bounds__(kT2, 1) kda_bwd_chain(BwdChunkArgs a)
{
    extern __shared__ __align__(16) float sm[];
    const int h = blockIdx.y, n = blockIdx.z, slice = blockIdx.x >> 1;
    if (a.seq_heads[h]) return;
    if (blockIdx.x & 1) chain_run<NS, true>(a, sm, n, h, slice * NS);
    else chain_run<NS, false>(a, sm, n, h, slice * NS);
}

}  // namespace

kda_status_t launch_bwd_chunk(const BwdChunkArgs& a, kda_dtype_t dt, int32_t* chunk_cu_dev, cudaStream_t st)
{
    {
        DeviceLock lk;
        if (!lk.st) return lk.rc;
        if (!lk.st->attr_done[15]) {
            const auto attr = cudaFuncAttributeMaxDynamicSharedMemorySize;
            KDA_CUDA_TRY(cudaFuncSetAttribute(kda_bwd_intra<float>, attr, (int)kSmem1));
            KDA_CUDA_TRY(cudaFuncSetAttribute(kda_bwd_intra<__nv_bfloat16>, attr, (int)kSmem1));
            KDA_CUDA_TRY(cudaFuncSetAttribute(kda_bwd_chain<64>, attr, (int)ChainSmem<64>::kBytes));
            KDA_CUDA_TRY(cudaFuncSetAttribute(kda_bwd_chain<32>, attr, (int)ChainSmem<32>::kBytes));
            lk.st->attr_done[15] = true;
        }
    }
    kda_bwd_prep<<<1, 256, 0, st>>>(a.hdr, a.cu_seqlens, chunk_cu_dev, a.n_seqs, a.seq_heads, a.H);
    const dim3 grid((unsigned)a.n_chunks, (unsigned)a.H);
    if (a.n_chunks > 0) {
        ProfScope ps(PROF_INTRA, st);
        if (dt == KDA_BF16) kda_bwd_intra<__nv_bfloat16><<<grid, kT1, kSmem1, st>>>(a);
        else kda_bwd_intra<float><<<grid, kT1, kSmem1, st>>>(a);
    }
    {
        ProfScope ps(PROF_INTER, st);
        // one CTA per SM (shared memory): 32-column slices only while they fit one wave
        const bool narrow = (int64_t)a.n_seqs * a.H * 8 <= 148;
        if (narrow) kda_bwd_chain<32><<<dim3(8, (unsigned)a.H, (unsigned)a.n_seqs), kT2, ChainSmem<32>::kBytes, st>>>(a);
        else kda_bwd_chain<64><<<dim3(4, (unsigned)a.H, (unsigned)a.n_seqs), kT2, ChainSmem<64>::kBytes, st>>>(a);
    }
    count_launch(a.n_chunks > 0 ? 3 : 2);
    KDA_CUDA_TRY(cudaGetLastError());
    return a.n_chunks > 0 ? launch_bwd_out(a, dt, st) : KDA_OK;
}

}  // namespace kda
