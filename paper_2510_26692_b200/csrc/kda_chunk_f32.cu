// fp32 path of the chunkwise KDA forward (paper Section 3.1; steps follow Appendix C's order), dt = KDA_F32.
// The products run on split tf32 operands (kda_mma3.cuh: 22 significant bits, step sums rounded to
// nearest; single tf32 or bf16 products could not meet the 1e-4 tolerance), everything else is fp32.
//
// Two kernels per pass over a range of chunks:
//   intra  one CTA per (chunk, head): cumulative log-decay G (a1), gated Gram matrices
//          StrictTril((Gamma.K)(K/Gamma)^T) (a2) and Aqk = Tril((Gamma.Q)(K/Gamma)^T) (a5),
//          T = (I + . Diag(beta))^-1 (a3; Diag(beta) T = (I + Akk)^-1 Diag(beta)), W = Diag(beta) T (Gamma.K),
//          U = Diag(beta) T V (a4).  Writes W, U, Gamma.Q, (gamma^C/Gamma).K, Aqk, gamma^C to a scratch tile.
//   inter  one CTA per (sequence, head, 8- or 16-column slice of dv), sequential over the chunks:
//          V_new = U - W S (a6), O = (Gamma.Q) S + Aqk V_new (a7),
//          S <- Diag(gamma^C) S + ((gamma^C/Gamma).K)^T V_new (a8).  State columns are independent,
//          which is what lets dv be sliced across CTAs.
//
// The decay ratios exp(G_i - G_j) are factored around G_m = G_C / 2 (per channel) as
// exp(G_i - G_m) * exp(G_m - G_j), with each exponent clamped to [-80, 80], so no product
// overflows fp32; entries above the diagonal are never used (selected to zero, not multiplied).
//
// A call of this path is small (256 tokens x 2 heads: eight tiles), so what bounds it is the length of a tile's
// chain of phases and of a chain step, not any throughput: 512 threads per tile, the substitution as
// blocks, the operands of a chain phase fetched during the other; a tile in three CTAs and a chain of 8 columns
// where SMs would be idle.  Measured at 256 tokens x 2 heads: 30.3 us a call (intra 17, inter 16, overlapping),
// 39.5 with one CTA per tile and 16 columns per chain, 104 us with FMA products and a substitution of one
// thread per column; 2048 tokens x 8 heads: 155 us, 185 before.
#include <type_traits>

#include "kda_common.cuh"
#include "kda_mma3.cuh"
#include "kda_ptx.cuh"

namespace kda {
namespace {

using namespace mma3;

constexpr float kClamp = 80.f;
// Below this chunk decay a factor exp(G - G_m) may be so small that its low tf32 part is denormal, which
// the tensor core flushes: the Gram matrices are then formed with FMA instructions.
constexpr float kSplitRange = -100.f;
constexpr int LR = 132, LC = 136, LM = 68;       // row pitches: k-contiguous, k-strided, 64 x 64

// scratch tile (floats)
constexpr int T_W = 0;
constexpr int T_U = T_W + kC * kD;
constexpr int T_QG = T_U + kC * kD;
constexpr int T_KT = T_QG + kC * kD;
constexpr int T_AQK = T_KT + kC * kD;
constexpr int T_GC = T_AQK + kC * kC;
constexpr int T_FLOATS = T_GC + kD;

// The log decay as a LogSum.  With its high part alone: error of o 2.1e-7 at a decay of sigmoid(4) a token but 7.2e-7 at
// sigmoid(-1); with both 2.0e-7 and 2.5e-7.
// (a NaN stays one: fminf and fmaxf would turn it into a bound)
__device__ __forceinline__ float clampf(float x) { return x == x ? fminf(fmaxf(x, -kClamp), kClamp) : x; }

constexpr int kT1 = 512;
namespace s1 {
constexpr int KG = 0;                            // K exp(G - G_m)          [64][LR]
constexpr int KI = KG + 64 * LR;                 // K exp(G_m - G)          [64][LR]
constexpr int QG = KI + 64 * LR;                 // scale Q exp(G - G_m)    [64][LR]
constexpr int V = QG + 64 * LR;                  // [64][LC]
constexpr int B = V + 64 * LC;                   // [64][LM]
constexpr int T = B + 64 * LM;                   // [64][LM]
constexpr int VEC = T + 64 * LM;                 // exp(G_m) [128], beta [64], segment sums [4][128] twice
constexpr int kFloats = VEC + 128 + 64 + 1024;
}  // namespace s1
constexpr size_t kSmem1 = (size_t)s1::kFloats * 4;
static_assert(kSmem1 <= 232448, "fits the shared memory of one SM");

template <bool whole>
__global__ void __launch_bounds__(kT1, 1) kda_intra_f32(ChunkArgs a, float* __restrict__ tiles, WsHeader* hdr)
{
    extern __shared__ __align__(16) float sm[];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const int h = blockIdx.y;
    const int64_t gc_idx = a.g0 + blockIdx.x;
    // a tile whole, or in three parts
    const bool part_w = whole || blockIdx.z == 0, part_u = whole || blockIdx.z == 1,
               part_q = whole || blockIdx.z == 2;
    ptx::grid_dep_wait();
    ptx::grid_dep_launch();
    const ChunkLoc loc = locate_chunk(a, gc_idx);
    const float* qp = static_cast<const float*>(a.q);
    const float* kp = static_cast<const float*>(a.k);
    const float* vp = static_cast<const float*>(a.v);
    float* tile = tiles + ((size_t)blockIdx.x * a.H + h) * T_FLOATS;
    float* sKG = sm + s1::KG; float* sKI = sm + s1::KI; float* sQG = sm + s1::QG; float* sV = sm + s1::V;
    float* sB = sm + s1::B; float* sT = sm + s1::T;
    float* sEm = sm + s1::VEC; float* sBeta = sEm + 128; float* sSeg = sBeta + 64;

    // a1: thread = channel c of 16 consecutive tokens (identity padding past the sequence end)
    const int c = t & 127, seg = t >> 7;
    float G[16], kk[16], qq[16];
    float z = 0.f;       // becomes a NaN with the first value that is not finite
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const int r = seg * 16 + i;
        const size_t off = ((size_t)(loc.tok0 + r) * a.H + h) * kD + c;
        const bool in = r < loc.len;
        G[i] = in ? a.log_alpha[off] : 0.f;
        kk[i] = in ? kp[off] : 0.f;
        qq[i] = in && qp && part_q ? qp[off] : 0.f;
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) z = fmaf(0.f, G[i], fmaf(0.f, kk[i], fmaf(0.f, qq[i], z)));
    for (int idx = part_u ? t : 64 * 32; idx < 64 * 32; idx += kT1) {
        const int r = idx >> 5, x = (idx & 31) * 4;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (r < loc.len) v = *reinterpret_cast<const float4*>(vp + ((size_t)(loc.tok0 + r) * a.H + h) * kD + x);
        *reinterpret_cast<float4*>(sV + r * LC + x) = v;
        z = fmaf(0.f, v.x, fmaf(0.f, v.y, fmaf(0.f, v.z, fmaf(0.f, v.w, z))));
    }
    if (t < 64) sBeta[t] = t < loc.len ? a.beta[(size_t)(loc.tok0 + t) * a.H + h] : 0.f;
    LogSum run = {0.f, 0.f};
#pragma unroll
    for (int i = 0; i < 16; ++i) run = run + G[i];
    sSeg[seg * 128 + c] = run.hi;
    sSeg[512 + seg * 128 + c] = run.lo;
    for (int idx = t; idx < 64 * LM; idx += kT1) sT[idx] = 0.f;
    if (t < 64) z = fmaf(0.f, sBeta[t], z);
    // A token that is not finite may spoil later tokens but no earlier ones: such a tile forms its products entry by
    // entry over the triangle, where a matrix instruction would multiply the zeros beside it.
    const int odd = __syncthreads_or(z != 0.f);
    LogSum g = {0.f, 0.f}, total = {0.f, 0.f};
#pragma unroll
    for (int s = 0; s < 4; ++s) {
        if (s == seg) g = total;
        total = total + sSeg[s * 128 + c];
        total.lo += sSeg[512 + s * 128 + c];
    }
    // a channel that decays by more than e^-160 inside the chunk leaves the range of the
    // two-factor form (the clamp keeps everything finite): flag the call
    if (total.hi < -2.f * kClamp) atomicOr(&hdr->flags, 1);
    const bool nan = total.hi != total.hi;
    const LogSum gm = {nan ? 0.f : 0.5f * total.hi, nan ? 0.f : 0.5f * total.lo};
    const float em = exp_of(gm);
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const int r = seg * 16 + i;
        g = g + G[i];
        LogSum x = g - gm;
        const float cut = clampf(x.hi);
        x = {cut, cut == x.hi ? x.lo : 0.f};
        const float e1 = exp_of(x), e2 = exp_of({-x.hi, -x.lo});
        sKG[r * LR + c] = kk[i] * e1;
        sKI[r * LR + c] = kk[i] * e2;
        if (part_q) {
            const float q1 = a.scale * qq[i] * e1;
            sQG[r * LR + c] = q1;
            tile[T_QG + r * kD + c] = q1 * em;
            tile[T_KT + r * kD + c] = kk[i] * exp_of(total - g);
        }
    }
    if (seg == 0) {
        sEm[c] = em;
        if (part_q) tile[T_GC + c] = exp_of(total);
    }
    const int far = __syncthreads_or(total.hi < kSplitRange) | odd;

    // a2 + a5: [K^ ; Q] K_^T: warps 4 x 4, 32 x 16 entries each of 128 rows, or 16 x 16 of 64; only blocks that
    // reach the triangle
    auto gram = [&](auto tag, bool is_q, int r0, int c0) {
        constexpr int MT = decltype(tag)::value;
        const float* A = (is_q ? sQG : sKG) + r0 * LR;
        float acc[MT][2][4];
        zero(acc);
        if (c0 < r0 + 16 * MT && (!is_q || qp)) {
            if (!far) {
                gemm<0, 2, false, true, false, false>(acc, A, LR, sKI + c0 * LR, LR, 0, kD, lane);
            } else {
                const int g = lane >> 2, c2 = 2 * (lane & 3);
                for (int k = 0; k < kD; ++k)
#pragma unroll
                    for (int m = 0; m < MT; ++m)
#pragma unroll
                        for (int n = 0; n < 2; ++n)
#pragma unroll
                            for (int j = 0; j < 4; ++j)
                                acc[m][n][j] = fmaf(A[(16 * m + g + 8 * (j >> 1)) * LR + k],
                                                    sKI[(c0 + 8 * n + c2 + (j & 1)) * LR + k], acc[m][n][j]);
            }
        }
        each_pair(acc, lane, [&](int i, int j, float x, float y) {
            i += r0; j += c0;
            if (!is_q) {
                st2(sB + i * LM + j, j < i ? x * sBeta[j] : 0.f, j + 1 < i ? y * sBeta[j + 1] : 0.f);
            } else {
                st2(tile + T_AQK + i * kC + j, j <= i ? x : 0.f, j + 1 <= i ? y : 0.f);
            }
        });
    };
    if (whole) gram(std::integral_constant<int, 2>{}, w >= 8, ((w >> 2) & 1) * 32, (w & 3) * 16);
    else gram(std::integral_constant<int, 1>{}, part_q, (w >> 2) * 16, (w & 3) * 16);
    if (!part_w && !part_u) return;
    __syncthreads();
    if (odd) {
        if (t < 64)
            for (int i = t; i < 64; ++i) {       // column t
                float x = i == t ? 1.f : 0.f;
                for (int m = t; m < i; ++m) x = fmaf(-sB[i * LM + m], sT[m * LM + t], x);
                sT[i * LM + t] = x;
            }
        __syncthreads();
        for (int idx = t; idx < 64 * kD; idx += kT1) {
            const int i = idx >> 7, x = idx & 127;
            float wi = 0.f, ui = 0.f;
            for (int j = 0; j <= i; ++j) {
                wi = fmaf(sT[i * LM + j], sKG[j * LR + x], wi);
                if (part_u) ui = fmaf(sT[i * LM + j], sV[j * LC + x], ui);
            }
            if (part_w) tile[T_W + idx] = sBeta[i] * wi * sEm[x];
            if (part_u) tile[T_U + idx] = sBeta[i] * ui;
        }
        return;
    }
    invert_unit_lower<LM>(sB, sT, t, [] { __syncthreads(); });      // a3

    // a4: warps 2 x 8, 32 x 16 entries each; the triangle bounds the sums
    {
        const int r0 = (w >> 3) * 32, c0 = (w & 7) * 16;
        float acc[2][2][4];
        zero(acc);
        if (part_w) gemm<0, 2, false, false, false, false>(acc, sT + r0 * LM, LM, sKG + c0, LR, 0, r0 + 32, lane);
        if (part_w) each_pair(acc, lane, [&](int i, int j, float x, float y) {
            const float b = sBeta[r0 + i];
            st2(tile + T_W + (r0 + i) * kD + c0 + j, b * x * sEm[c0 + j], b * y * sEm[c0 + j + 1]);
        });
        if (!part_u) return;
        zero(acc);
        gemm<0, 2, false, false, false, false>(acc, sT + r0 * LM, LM, sV + c0, LC, 0, r0 + 32, lane);
        each_pair(acc, lane, [&](int i, int j, float x, float y) {
            const float b = sBeta[r0 + i];
            st2(tile + T_U + (r0 + i) * kD + c0 + j, b * x, b * y);
        });
    }
}

constexpr int kT2 = 256;
template <int NS> struct s2 {                           // NS = dv columns per inter-chunk CTA
    static constexpr int LS = NS == 8 ? 8 : NS + 8;
    static constexpr int W = 0;                 // [64][LR]   operands of the first phase: W, Gamma.Q, U
    static constexpr int Q = W + 64 * LR;       // [64][LR]
    static constexpr int U = Q + 64 * LR;       // [64][LS]
    static constexpr int KT = U + 64 * LS;      // [64][LC]   operands of the second: (gamma^C/Gamma).K, Aqk
    static constexpr int A = KT + 64 * LC;      // [64][LM]
    static constexpr int S = A + 64 * LM;       // [128][LS]  state
    static constexpr int VN = S + 128 * LS;     // [64][LS]   V_new
    static constexpr size_t kBytes = (size_t)(VN + 64 * LS) * 4;
};

// Eight warps of 16 rows each.  First phase: [W ; Gamma.Q] S (128 rows); second: Aqk V_new into the output rows
// of warps 4-7, and the state's 128 rows, which stay in the accumulator fragments of all warps (copy in
// shared memory as B operand).  The operands of each phase arrive by cp.async during the other.
template <int NS>
__global__ void __launch_bounds__(kT2, 1) kda_inter_f32(ChunkArgs a, const float* tiles, int n_begin)
{
    using L = s2<NS>;
    constexpr int LS = L::LS, NT = NS / 8;
    extern __shared__ __align__(16) float sm[];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5, g = lane >> 2;
    const int h = blockIdx.y, n = n_begin + blockIdx.z;
    const int col0 = blockIdx.x * NS;
    float* op = static_cast<float*>(a.o);
    ptx::grid_dep_wait();
    ptx::grid_dep_launch();

    int64_t cb, ce, tok_begin, tok_end;
    if (a.cu_seqlens) {
        cb = a.chunk_cu[n]; ce = a.chunk_cu[n + 1];
        tok_begin = a.cu_seqlens[n]; tok_end = a.cu_seqlens[n + 1];
    } else {
        cb = (int64_t)n * a.chunks_per_seq; ce = cb + a.chunks_per_seq;
        tok_begin = (int64_t)n * a.seq_len; tok_end = tok_begin + a.seq_len;
    }
    const int64_t seq_c0 = cb;
    if (cb < a.g0) cb = a.g0;
    if (ce > a.g1) ce = a.g1;

    auto tile_of = [&](int64_t c) { return tiles + ((size_t)(c - a.g0) * a.H + h) * T_FLOATS; };
    auto fetch1 = [&](int64_t ch) {
        const float* tile = tile_of(ch);
        for (int idx = t; idx < 64 * 32; idx += kT2) {
            const int r = idx >> 5, x = (idx & 31) * 4;
            cp16(sm + L::W + r * LR + x, tile + T_W + r * kD + x);
            if (op) cp16(sm + L::Q + r * LR + x, tile + T_QG + r * kD + x);
        }
        for (int idx = t; idx < 64 * (NS / 4); idx += kT2) {
            const int r = idx / (NS / 4), x = idx % (NS / 4) * 4;
            cp16(sm + L::U + r * LS + x, tile + T_U + r * kD + col0 + x);
        }
        cp_commit();
    };
    auto fetch2 = [&](int64_t ch) {
        const float* tile = tile_of(ch);
        for (int idx = t; idx < 64 * 32; idx += kT2) {
            const int r = idx >> 5, x = (idx & 31) * 4;
            cp16(sm + L::KT + r * LC + x, tile + T_KT + r * kD + x);
        }
        if (op)
            for (int idx = t; idx < 64 * 16; idx += kT2) {
                const int r = idx >> 4, x = (idx & 15) * 4;
                cp16(sm + L::A + r * LM + x, tile + T_AQK + r * kC + x);
            }
        cp_commit();
    };

    if (cb < ce) { fetch1(cb); fetch2(cb); }
    const size_t sbase = ((size_t)n * a.H + h) * (size_t)(kD * kD) + col0;
    float* sS = sm + L::S;
    float* sVn = sm + L::VN;
    float S[1][NT][4];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int hf = 0; hf < 2; ++hf) {
            const int r = 16 * w + 8 * hf + g, x = 8 * nt + 2 * (lane & 3);
            float2 v = make_float2(0.f, 0.f);
            if (a.S_in) v = *reinterpret_cast<const float2*>(a.S_in + sbase + (size_t)r * kD + x);
            S[0][nt][2 * hf] = v.x; S[0][nt][2 * hf + 1] = v.y;
            st2(sS + r * LS + x, v.x, v.y);
        }
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    __syncthreads();
    for (int64_t ch = cb; ch < ce; ++ch) {
        const float* tile = tile_of(ch);
        const float gam0 = tile[T_GC + 16 * w + g], gam1 = tile[T_GC + 16 * w + 8 + g];
        float acc[1][NT][4];
        zero(acc);
        if (w < 4 || op)
            gemm<0, NT, false, false, false, false>(acc, sm + (w < 4 ? L::W + 16 * w * LR : L::Q + 16 * (w - 4) * LR), LR, sS,
                                                   LS, 0, kD, lane);
        float z = 0.f;
        if (w < 4)
            each_pair(acc, lane, [&](int i, int j, float x, float y) {
                const float2 u = *reinterpret_cast<const float2*>(sm + L::U + (16 * w + i) * LS + j);
                st2(sVn + (16 * w + i) * LS + j, u.x - x, u.y - y);
                z = fmaf(0.f, u.x - x, fmaf(0.f, u.y - y, z));
            });
        cp_wait0();
        const int odd = __syncthreads_or(z != 0.f);     // (V_new not finite: see kda_intra_f32)
        if (ch + 1 < ce) fetch1(ch + 1);
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
            S[0][nt][0] *= gam0; S[0][nt][1] *= gam0;
            S[0][nt][2] *= gam1; S[0][nt][3] *= gam1;
        }
        gemm<0, NT, true, false, false, false>(S, sm + L::KT + 16 * w, LC, sVn, LS, 0, kC, lane);
        each_pair(S, lane, [&](int i, int j, float x, float y) { st2(sS + (16 * w + i) * LS + j, x, y); });
        if (w >= 4 && op) {
            const int r0 = 16 * (w - 4);
            if (!odd)
                gemm<0, NT, false, false, false, false>(acc, sm + L::A + r0 * LM, LM, sVn, LS, 0, r0 + 16, lane);
            else
                for (int nt = 0; nt < NT; ++nt)
                    for (int e = 0; e < 4; ++e) {
                        const int row = r0 + g + 8 * (e >> 1), x = 8 * nt + 2 * (lane & 3) + (e & 1);
                        float s = acc[0][nt][e];
                        for (int j = 0; j <= row; ++j) s = fmaf(sm[L::A + row * LM + j], sVn[j * LS + x], s);
                        acc[0][nt][e] = s;
                    }
            const int64_t tok0 = tok_begin + (ch - seq_c0) * kC;
            each_pair(acc, lane, [&](int i, int j, float x, float y) {
                const int64_t tok = tok0 + r0 + i;
                if (tok < tok_end) st2(op + ((size_t)tok * a.H + h) * kD + col0 + j, x, y);
            });
        }
        cp_wait0();
        __syncthreads();
        if (ch + 1 < ce) fetch2(ch + 1);
    }
    each_pair(S, lane, [&](int i, int j, float x, float y) { st2(a.S_out + sbase + (size_t)(16 * w + i) * kD + j, x, y); });
}

__global__ void kda_prep_kernel(WsHeader* hdr, const int32_t* cu, int32_t* chunk_cu, int n_seqs)
{
    ptx::grid_dep_wait();        // (launched before the preceding kernel has ended)
    ptx::grid_dep_launch();
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        hdr->status = 0;
        hdr->where = 0;
        hdr->flags = 0;
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

size_t f32_tile_bytes() { return (size_t)T_FLOATS * sizeof(float); }

kda_status_t launch_chunk_f32(const ChunkArgs& a, void* tiles, int n_begin, int n_count, WsHeader* hdr, cudaStream_t st)
{
    int n_sm = 0;
    {
        DeviceLock lk;
        if (!lk.st) return lk.rc;
        if (!lk.st->attr_done[4]) {
            KDA_CUDA_TRY(cudaFuncSetAttribute(kda_intra_f32<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem1));
            KDA_CUDA_TRY(cudaFuncSetAttribute(kda_intra_f32<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem1));
            KDA_CUDA_TRY(cudaFuncSetAttribute(kda_inter_f32<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)s2<8>::kBytes));
            KDA_CUDA_TRY(cudaFuncSetAttribute(kda_inter_f32<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)s2<16>::kBytes));
            lk.st->attr_done[4] = true;
        }
        if (lk.st->n_sm == 0) {
            int dev = 0;
            KDA_CUDA_TRY(cudaGetDevice(&dev));
            KDA_CUDA_TRY(cudaDeviceGetAttribute(&lk.st->n_sm, cudaDevAttrMultiProcessorCount, dev));
        }
        n_sm = lk.st->n_sm;
    }
    if (n_count > 65535)
        return fail(KDA_ERR_UNSUPPORTED, "kda_chunk_fwd: more than 65535 sequences in one fp32 call");
    const int64_t n_chunks = a.g1 - a.g0;
    float* tp = static_cast<float*>(tiles);
    if (n_chunks > 0) {
        ProfScope ps(PROF_INTRA, st);
        // three CTAs per tile (W; U; Aqk and what is only gated) while there are SMs for all: each repeats the
        // gating, and W and U the Gram matrix and its inverse, so more of them cost work but no time
        const bool parts = n_chunks * a.H * 3 <= n_sm;
        KDA_CUDA_TRY(launch_dependent(parts ? kda_intra_f32<false> : kda_intra_f32<true>,
                                      dim3((unsigned)n_chunks, (unsigned)a.H, parts ? 3 : 1), kT1, kSmem1, st, a, tp, hdr));
        count_launch();
    }
    if (n_count > 0) {
        ProfScope ps(PROF_INTER, st);
        const dim3 grid16(kD / 16, (unsigned)a.H, (unsigned)n_count), grid8(kD / 8, (unsigned)a.H, (unsigned)n_count);
        // a chain step is a latency, shorter for fewer columns: 8 as long as those CTAs have an SM each
        if ((int64_t)(kD / 8) * a.H * n_count <= n_sm)
            KDA_CUDA_TRY(launch_dependent(kda_inter_f32<8>, grid8, kT2, s2<8>::kBytes, st, a, (const float*)tp, n_begin));
        else
            KDA_CUDA_TRY(launch_dependent(kda_inter_f32<16>, grid16, kT2, s2<16>::kBytes, st, a, (const float*)tp, n_begin));
        count_launch();
    }
    return KDA_OK;
}

kda_status_t launch_prep(WsHeader* hdr, const int32_t* cu_seqlens, int32_t* chunk_cu, int n_seqs,
                         cudaStream_t st)
{
    ProfScope ps(PROF_PREP, st);
    KDA_CUDA_TRY(launch_dependent(kda_prep_kernel, dim3(1), 32, 0, st, hdr, cu_seqlens, chunk_cu, n_seqs));
    count_launch();
    return KDA_OK;
}

}  // namespace kda
