// What the translation units of the backward pass share: the arguments and the per-(chunk, head)
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
    int* seq_heads;   // [H]: 1 = a chunk of this head decays too fast for the chunkwise form, or a token is not finite
    int n_seqs, H;
    WsHeader* hdr;
    int64_t seq_len, chunks_per_seq, n_chunks;
    float scale;
    unsigned long long wait_limit_ns;
    int n_sm;
};

// Scratch tile (floats), written by the first kernel unless stated otherwise.  K^, K_ and Q are relative to the
// middle G_m of the chunk's log decay (K^ = k e^(G - G_m), K_ = k e^(G_m - G)); the chains restore the true
// scale on the state.  "rf" = rows fastest: element (row, c) of a matrix with R rows at float
// ((c / 4) R + row) 4 + c % 4, which a thread per row reads and writes in whole 16-byte pieces beside its
// neighbours'.  What the chains read and write has the columns of the state in the rows, as they have them in the TMEM
// lanes; the states that they leave have its rows there (sf), as the gradients stage needs them.
namespace bt {
constexpr int WI = 0;                // W'^T [128][64] as a split image (kda_split3.cuh), W' = T' K^, T' = (I + B Diag(beta))^-1
constexpr int KI = WI + 12288;       // K_ [64][128] as a split image
constexpr int R = KI + 12288;        // [128][64] rf: U'^T, U' = T' V, replaced by r^T, r = U' - W' S, by the forward chain
constexpr int X = R + 64 * 128;      // [128][64] rf: dO^T P, replaced by dX^T, dX = P^T dO + K~ Lam, by the backward chain
constexpr int N = X + 64 * 128;      // [128][128] rf: dO^T Q
constexpr int kState = 128 * 128;
constexpr int S = N + 128 * 128;     // [128][128] sf: state entering the chunk (forward chain)
constexpr int L = S + kState;        // [128][128] sf: adjoint of the state leaving the chunk (backward chain)
constexpr int F = L + kState;        // [64][128] e^(G - G_m)
constexpr int T = F + 64 * 128;      // [64][64] T'
constexpr int B = T + 64 * 64;       // [64][64] B = StrictTril(K^ K_^T)
constexpr int GC = B + 64 * 64;      // [128] e^(G_C)
constexpr int EM = GC + 128;         // [128] e^(G_m), also e^(G_C - G_m)
constexpr int BE = EM + 128;         // [64] beta, zero past the end of the sequence
constexpr int kFloats = BE + 64;
constexpr int kVec = kFloats - GC;   // the vectors
}  // namespace bt
__device__ __forceinline__ int rf(int rows, int row, int c) { return ((c >> 2) * rows + row) * 4 + (c & 3); }
// rf of 128 rows with the rows of a group of four columns in another order from group to group: a warp with the columns in its
// lanes writes a row to shared memory without bank conflicts
__device__ __forceinline__ int sf(int row, int c) { return (c >> 2) * 512 + ((row ^ ((c >> 2) & 7)) << 2) + (c & 3); }

// Largest decay of a chunk taken in chunk form.
constexpr float kBwdRange = 40.f;

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

// The per-chunk kernels hold one CTA per SM whose loads, products and stores take turns, so HBM idles while
// the tensor core works and the other way round.  Each CTA therefore asks for the tile n_sm places further on
// (likely the next on its SM) to come into L2 while it works itself: 148 tiles are 45 MB of the 126 MB.
__device__ __forceinline__ void prefetch_l2(const void* p, uint32_t bytes) {   // 16-byte aligned, multiple of 16
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}
// The rows of a chunk in token-major tensors, a 128-byte piece a thread and step (a row each by bulk prefetches, 64 threads
// issued 320 of them one after the other and held up the CTA's first barrier: the first stage 317 -> 285 us at 4096 x 32
// heads, the gradients 458 -> 415).
template <int kThreads, typename T, int kN>
__device__ __forceinline__ void prefetch_rows(const BwdLoc& l, int H, int h, int t, const T* const (&p)[kN]) {
    constexpr int kLines = kD * (int)sizeof(T) / 128;
#pragma unroll
    for (int i = 0; i < kN; ++i)
        if (p[i])
            for (int x = t; x < l.len * kLines; x += kThreads)
                asm volatile("prefetch.global.L2 [%0];" ::"l"(reinterpret_cast<const char*>(p[i] + ((size_t)(l.tok0 + x / kLines) * H + h) * kD) +
                                                                 (x % kLines) * 128));
}
// Tiles in the order of memory, heads fastest: the CTAs that run together then read and write whole rows of
// the token-major tensors (a head's share of a row is 256 or 512 bytes).
__device__ __forceinline__ void bwd_tile(const BwdChunkArgs& a, int64_t id, int64_t& g, int& h) {
    g = (int64_t)((uint32_t)id / (uint32_t)a.H);
    h = (int)(id - g * a.H);
}
// the tile n_sm places behind tile `id`; false if there is none
__device__ __forceinline__ bool bwd_next(const BwdChunkArgs& a, int64_t id, int64_t& g, int& h) {
    id += a.n_sm;
    if (id >= a.n_chunks * a.H) return false;
    bwd_tile(a, id, g, h);
    return true;
}

// 1 / x of a factor e^(+-20), one instruction (at most one unit in the last place off)
__device__ __forceinline__ float reciprocal(float x) {
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// Eight consecutive elements as they are stored.  The loads are volatile so that they stay where they are
// written, ahead of the stores and waits that they overlap; `in` = false gives zeros.
template <typename T> struct Raw8 { uint32_t w[2 * sizeof(T)]; };
__device__ __forceinline__ void ldraw4(uint32_t* w, const void* p) {
    asm volatile("ld.global.nc.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "l"(p));
}
// the same for data that this kernel itself overwrites later
__device__ __forceinline__ void ldraw4_w(uint32_t* w, const void* p) {
    asm volatile("ld.global.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "l"(p) : "memory");
}
__device__ __forceinline__ void ldraw(Raw8<float>& r, const float* p, bool in = true) {
#pragma unroll
    for (int e = 0; e < 8; ++e) r.w[e] = 0u;
    if (in) { ldraw4(r.w, p); ldraw4(r.w + 4, p + 4); }
}
__device__ __forceinline__ void ldraw(Raw8<__nv_bfloat16>& r, const __nv_bfloat16* p, bool in = true) {
#pragma unroll
    for (int e = 0; e < 4; ++e) r.w[e] = 0u;
    if (in) ldraw4(r.w, p);
}
__device__ __forceinline__ void to_f(const Raw8<float>& r, float (&x)[8]) {
#pragma unroll
    for (int e = 0; e < 8; ++e) x[e] = __uint_as_float(r.w[e]);
}
__device__ __forceinline__ void to_f(const Raw8<__nv_bfloat16>& r, float (&x)[8]) {
#pragma unroll
    for (int e = 0; e < 4; ++e) { x[2 * e] = __uint_as_float(r.w[e] << 16); x[2 * e + 1] = __uint_as_float(r.w[e] & 0xffff0000u); }
}

// Whether a value that the split images (kda_split3.cuh) cannot hold is among those looked at: not finite, or
// rounded to an infinity as a bf16 number.
__device__ __forceinline__ void look(uint32_t& seen, const Raw8<float>& r) {
#pragma unroll
    for (int e = 0; e < 8; ++e) seen |= (r.w[e] & 0x7fffffffu) + 0x00808000u;
}
__device__ __forceinline__ void look(uint32_t& seen, const Raw8<__nv_bfloat16>& r) {
#pragma unroll
    for (int e = 0; e < 4; ++e) seen |= (r.w[e] & 0x7f807f80u) + 0x00800080u;
}
template <typename T> __device__ __forceinline__ bool seen_odd(uint32_t seen) {
    return (seen & (sizeof(T) == 4 ? 0x80000000u : 0x80008000u)) != 0u;
}

kda_status_t launch_bwd_intra(const BwdChunkArgs& a, kda_dtype_t dt, cudaStream_t st);
kda_status_t launch_bwd_chain(const BwdChunkArgs& a, cudaStream_t st);
kda_status_t launch_bwd_out(const BwdChunkArgs& a, kda_dtype_t dt, cudaStream_t st);
kda_status_t launch_bwd_chunk(BwdChunkArgs a, kda_dtype_t dt, int32_t* chunk_cu_dev, cudaStream_t st);

}  // namespace kda
