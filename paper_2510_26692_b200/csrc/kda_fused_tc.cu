// bf16 tensor-core path of the chunkwise KDA forward (paper Section 3.1; Appendix C): two stages, either as two
// kernels (kda_intra_tc over all tiles, then kda_chain_tc, a CTA per chain) or as one (kda_fused_tc: thread-block
// clusters of one chain CTA and two or three engine CTAs).  CTAs of 512 threads run warp-specialised roles that meet
// only on mbarriers and named barriers, those of a cluster on mbarriers in distributed shared memory:
//
//   intra-chunk engine (8 warps, two to a CTA): everything of a (chunk, head) tile that does not depend on the state --
//     a1   G = cumulative sum of log alpha over the chunk's tokens (fp32, log2 domain)
//          gated operands, bf16:  Kg = K exp(G - G_m),  Qg = scale Q exp(G - G_m),  Ki = K exp(G_m - G)
//          with G_m = G_C / 2 per channel (the middle of the chunk's log-decay range), so that
//          exp(G_i - G_j) = exp(G_i - G_m) exp(G_m - G_j) is formed from two factors of bounded range.  G_m is taken
//          as a whole number of halvings: W and Q get their true scale exp(G_m) without another rounding, and the
//          rounding of Qg is the same in Aqk and in Q S.  (Rounded a second time: error of o 0.2 per cent larger at
//          a decay of sigmoid(4) a token, 1 per cent at sigmoid(6).)
//     a2/a5  one tcgen05 MMA group  [Kg ; Qg] (128 x 128)  x  Ki^T (128 x 64)  ->  TMEM:
//          L = Diag(beta) StrictTril(rows 0-63) (fp32),  Aqk = Tril(rows 64-127) (bf16)
//     a3   T = (I + L)^-1 by blocked forward substitution: 16x16 diagonal blocks column by column in
//          fp32 registers, sub-diagonal blocks as warp-level 16x16 products (mma.sync, tf32 inputs)
//     a4   Mm = T Diag(beta) (bf16);  second MMA group  [Mm ; Mm] x [Kg | V]  ->  W' = Mm Kg, U = Mm V
//   The tile (operand images of kda_tiles.cuh) goes to global memory; in the fused kernel to a ring of a few tiles per
//   engine that stays in L2.
//   Two kernels: 7.7 us a tile with two in flight per SM, where reading its inputs and writing it takes 7.2 at the copy
//   bandwidth.  Fused 9 (without outputs 7.5): the chain of its phases, of which shared memory lets no third one overlap, and
//   the shared memory itself.
//
//   inter-chunk chain (a CTA; roles and products: see chain_run): all 128 columns of the state of one (sequence,
//   head), walked over the chunks in order -- a6 V_new = U - W S, a8 the state, a7 the outputs.  1.02 us a step for
//   the final state alone, 1.2 with outputs: two dependent round trips tensor core - registers - tensor core.
//   Tiles arrive by 1-D bulk copies (TMA engine).
//
// Every wait (mbarrier, flag word) is bounded by a wall-clock limit; when one runs out the role
// records KDA_ERR_TIMEOUT in the workspace header, marks the call as aborted so that every other
// waiter of the call returns at once, drains its own copies and leaves; TMEM is freed at the end.
// Tail chunks: rows past the sequence end behave as identity steps (log alpha = 0, beta = 0,
// k = q = v = 0).
#include <cuda.h>

#include "kda_common.cuh"
#include "kda_ptx.cuh"
#include "kda_tiles.cuh"

namespace kda {
namespace {

constexpr int kThreads = 512;
constexpr int kEngThreads = 256;
// Lane 0 of an engine's warp 7 issues every bulk copy, finds the tiles and talks to the chain (warps 0 and 2 issue
// the MMAs); what it can it does during the blocked substitution, which warps 6 and 7 have no part in.
constexpr int kServiceThread = 224;
constexpr int LDT = 68;                                   // padded fp32 row of the 64x64 matrix
constexpr int LDD = 20;                                   // padded fp32 row of a 16x16 diagonal block
constexpr float kLog2e = 1.4426950408889634f;
constexpr float kClamp2 = 80.f * 1.4426950408889634f;     // the +-80 clamp in the log2 domain
constexpr float kClampX = kClamp2 + 0.5f;                 // (G_m is rounded to a whole number)

// Optional role timing (compile with -DKDA_FUSED_TIMING): one thread per role accumulates the
// nanoseconds spent between marks and adds them to the header's spare words at the end.
#ifdef KDA_FUSED_TIMING
#define KT_DECL(n) uint64_t kt_last_ = ptx::globaltimer_ns(); uint32_t kt_acc_[n] = {0}
#define KT_MARK(cond, slot) do { if (cond) { const uint64_t now_ = ptx::globaltimer_ns(); kt_acc_[slot] += (uint32_t)(now_ - kt_last_); kt_last_ = now_; } } while (0)
#define KT_FLUSH(cond, hdr, base, n) do { if (cond) { for (int s_ = 0; s_ < n; ++s_) atomicAdd(&(hdr)->pad[(base) + s_], (int)(kt_acc_[s_] >> 4)); } } while (0)
#else
#define KT_DECL(n) do {} while (0)
#define KT_MARK(cond, slot) do {} while (0)
#define KT_FLUSH(cond, hdr, base, n) do {} while (0)
#endif

// ---- shared-memory map of one engine (bytes from a 1024-aligned base) ------------------------------
constexpr uint32_t E_KQ = 0;            // [2 K-halves][128 rows][64] bf16: rows 0-63 Kg, 64-127 Qg
constexpr uint32_t E_KQ_HALF = 16384;
constexpr uint32_t E_AQ = E_KQ + 8192;  // Aqk image [64][64] bf16: over rows 64-127 of the first K-half (Q' has left by then)
constexpr uint32_t E_KI = 32768;        // Ki [2 K-halves][64][64] bf16; then Mm [128][64]; then the W' staging
constexpr uint32_t E_KI_HALF = 8192;
constexpr uint32_t E_V = 49152;         // V [2 column blocks][64 tokens][64] bf16 (token-major)
constexpr uint32_t E_V_BLOCK = 8192;
constexpr uint32_t E_A = 65536;         // fp32 [64][LDT]: L, X below the diagonal, T above it (transposed block
                                        // positions); then the U^T staging
constexpr uint32_t E_TD = E_A + 64 * LDT * 4;     // fp32 4 x [16][LDD]: diagonal blocks of T; scan exchange [8][128] before
constexpr uint32_t E_TD_BYTES = 4 * 16 * LDD * 4;
constexpr uint32_t E_BETA = E_TD + E_TD_BYTES;    // 64 fp32
constexpr uint32_t E_DESC = E_BETA + 256;         // three tile descriptors: this tile, the next, the one after
constexpr uint32_t E_CUR = E_DESC + 192;          // the service thread's EngineCursor
constexpr int kMaxDepth = FusedArgs::kMaxDepth;   // ring positions of an engine
constexpr uint32_t E_BAR = E_CUR + 64;          // 8-byte words: mma barrier, K barrier, abort word, Q barrier,
                                                  // (first engine) TMEM slot, V barrier
constexpr uint32_t E_KS = (E_BAR + 96 + 1023) / 1024 * 1024;   // raw k of the NEXT tile [2 K-halves][64][64] bf16
constexpr uint32_t E_NORM = E_KS + 16384;         // layer mode: 1 / |k_i|, 1 / |q_i| (64 fp32 each)
constexpr uint32_t E_GV = E_NORM + 512;           // gamma^C and exp(G_C - G_m) on their way to the tile
constexpr uint32_t E_EM = E_GV + tc::GV_BYTES;    // exp(G_m)
constexpr uint32_t E_BYTES = (E_EM + 512 + 1023) / 1024 * 1024;
static_assert(E_TD_BYTES >= 8 * 128 * 4 && E_TD_BYTES >= 4 * 16 * LDD * 4, "scan exchange and diagonal blocks fit");

// ---- shared-memory map of a chain CTA (bytes from the 1024-aligned base) -----------------------------
// Two rings: [W ; Q] is free again once the first product of its chunk is complete, the rest of the tile half a step
// later; the output block has a buffer of its own (kept over the [W ; Q] image of a three-stage ring of whole
// tiles, it held the stage back: 1.73 instead of 1.5 us a step).
constexpr int kStagesA = 2, kStagesB = 3;
constexpr uint32_t kABytes = 32768, kBBytes = tc::TILE_BYTES - tc::OFF_KI;   // B: K', Aqk, gate vectors, U^T
constexpr uint32_t C_STAGEB = (kBBytes + 1023) / 1024 * 1024;
constexpr uint32_t C_A = 0, C_B = kStagesA * kABytes;
constexpr uint32_t C_OUT = C_B + kStagesB * C_STAGEB;   // output block: [2][64 tokens][64] bf16, or 64 rows in fp32
constexpr uint32_t C_BAR = C_OUT + 32768;
constexpr uint32_t C_BYTES = C_BAR + 512;
// offsets inside a B stage
constexpr uint32_t B_KI = 0, B_AQ = tc::OFF_AQ - tc::OFF_KI, B_GV = tc::OFF_GV - tc::OFF_KI, B_U = tc::OFF_U - tc::OFF_KI;
constexpr uint32_t kSmemBytes = 2 * E_BYTES > C_BYTES ? 2 * E_BYTES : C_BYTES;
static_assert(E_BYTES % 1024 == 0, "operand images stay 1024-byte aligned");
static_assert(kSmemBytes <= 232448, "fits the shared memory of one SM");
// Registers of the chain kernel's compute warps: the fp32 state takes 64 of them, an accumulator another 32 (at 128, the
// share of each of 512 threads, some spilled: 1.33 instead of 1.25 us a step then).  The other half of the warps gives up as many.
constexpr int kChainRegs = 160;
constexpr uint32_t kTmemCols = 512;                // two engines of 256 columns, or one chain
// TMEM columns of a chain: D1 of two chunks, D3, the bf16 state and V_new (A operands, two values a column)
constexpr uint32_t T_D1 = 0, T_D3 = 256, T_S = 384, T_VN = 448;

// loads that the compiler may not sink below their issue point (register prefetch of the next tile)
__device__ __forceinline__ void ld_f4(const float* p, float& a, float& b, float& c, float& d) {
    asm volatile("ld.global.L1::no_allocate.v4.f32 {%0,%1,%2,%3}, [%4];"
                 : "=f"(a), "=f"(b), "=f"(c), "=f"(d)
                 : "l"(p));
}
// rounding to tf32 (to nearest, ties away) by an addition on the bit pattern: the tensor core ignores the 13 low
// bits (cvt.rna.tf32 gives the same and issues several times slower)
__device__ __forceinline__ uint32_t to_tf32(float x) { return __float_as_uint(x) + 0x1000u; }
// 16x16 block products of the forward substitution on the warp-level tensor path (mma.sync
// m16n8k8, tf32 inputs rounded to nearest, fp32 accumulation): acc += A * B with A, B 16x16 fp32
// blocks in shared memory (row strides lda, ldb floats).
__device__ __forceinline__ void block16_mma(float (&acc)[2][4], const float* pa, int lda, const float* pb,
                                            int ldb, int lane) {
    const int g = lane >> 2, t4 = lane & 3;
#pragma unroll
    for (int ks = 0; ks < 2; ++ks) {
        const uint32_t a0 = to_tf32(pa[g * lda + ks * 8 + t4]);
        const uint32_t a1 = to_tf32(pa[(g + 8) * lda + ks * 8 + t4]);
        const uint32_t a2 = to_tf32(pa[g * lda + ks * 8 + t4 + 4]);
        const uint32_t a3 = to_tf32(pa[(g + 8) * lda + ks * 8 + t4 + 4]);
#pragma unroll
        for (int nt = 0; nt < 2; ++nt) {
            const uint32_t b0 = to_tf32(pb[(ks * 8 + t4) * ldb + nt * 8 + g]);
            const uint32_t b1 = to_tf32(pb[(ks * 8 + t4 + 4) * ldb + nt * 8 + g]);
            asm volatile(
                "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
                "{%8,%9}, {%0,%1,%2,%3};"
                : "+f"(acc[nt][0]), "+f"(acc[nt][1]), "+f"(acc[nt][2]), "+f"(acc[nt][3])
                : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
        }
    }
}
__device__ __forceinline__ void block16_load(float (&acc)[2][4], const float* pc, int ld, int lane) {
    const int g = lane >> 2, t4 = lane & 3;
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) {
        const float2 lo = *reinterpret_cast<const float2*>(pc + g * ld + nt * 8 + 2 * t4);
        const float2 hi = *reinterpret_cast<const float2*>(pc + (g + 8) * ld + nt * 8 + 2 * t4);
        acc[nt][0] = lo.x; acc[nt][1] = lo.y; acc[nt][2] = hi.x; acc[nt][3] = hi.y;
    }
}
__device__ __forceinline__ void block16_store(float* pc, const float (&acc)[2][4], float sign, int ld,
                                              int lane) {
    const int g = lane >> 2, t4 = lane & 3;
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) {
        *reinterpret_cast<float2*>(pc + g * ld + nt * 8 + 2 * t4) =
            make_float2(sign * acc[nt][0], sign * acc[nt][1]);
        *reinterpret_cast<float2*>(pc + (g + 8) * ld + nt * 8 + 2 * t4) =
            make_float2(sign * acc[nt][2], sign * acc[nt][3]);
    }
}
__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ float lg2(float x) {
    float y;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// two values of an array as one operand of the packed fp32 operations (half the instructions of single ones)
__device__ __forceinline__ float2 pair(const float* x) { return make_float2(x[0], x[1]); }
__device__ __forceinline__ float2 both(float x) { return make_float2(x, x); }
__device__ __forceinline__ void set(float* x, float2 v) { x[0] = v.x; x[1] = v.y; }
__device__ __forceinline__ uint32_t pack_bf16(float a, float b);
__device__ __forceinline__ uint32_t pack_bf16(float2 v) { return pack_bf16(v.x, v.y); }
__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
    __nv_bfloat162 p = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<uint32_t*>(&p);
}

// ---- jobs: (sequence, head) pairs, dealt out to the clusters ------------------------------------------
struct JobInfo {
    int n, h, nch;
    int64_t tok_begin, tok_end;
    int64_t tile0;                // two-kernel schedule: index of the first tile (then every H-th)
};
// A run of a call cut into segments (kda_segments.cu).  kSeg: 0 = not cut, 1 = runs that find the segments' maps,
// 2 = runs from the states found.  Compiled apart: decided at run time it cost the whole chains 1 to 2 per cent.
struct SegInfo {
    int chain, p;                 // segment p of this chain
    bool unit;                    // its linear part: from the identity, without U
};
template <int kSeg>
__device__ __forceinline__ SegInfo seg_info(const FusedArgs& f, int id) {
    if (kSeg == 0) return {id, 0, false};
    const int runs = kSeg == 1 ? f.seg_runs : f.seg_P;
    const int s = id % runs;
    const bool unit = kSeg == 1 && s >= f.seg_val;
    return {id / runs, unit ? s - f.seg_val + 1 : s, unit};
}
// The state that a job starts from (nullptr = zero, or the identity) and the place of its final state (nullptr = not
// wanted).
template <int kSeg>
__device__ __forceinline__ const float* state_in(const FusedArgs& f, size_t off, int id) {
    const SegInfo s = seg_info<kSeg>(f, id);
    if (kSeg && s.p > 0) return kSeg == 1 ? nullptr : f.seg_scratch + ((size_t)s.chain * f.seg_runs + s.p - 1) * (kD * kD);
    return f.a.S_in ? f.a.S_in + off : nullptr;
}
template <int kSeg>
__device__ __forceinline__ float* state_out(const FusedArgs& f, size_t off, int id) {
    if (kSeg == 1) return f.seg_scratch + (size_t)id * (kD * kD);
    if (kSeg == 2 && seg_info<2>(f, id).p + 1 < f.seg_P) return nullptr;
    return f.a.S_out ? f.a.S_out + off : nullptr;
}
// Job number r of cluster cid (fused_job; sequences by f.order); false past its last.
__device__ __forceinline__ bool job_info(const FusedArgs& f, int cid, int r, JobInfo& I) {
    const int64_t jr = fused_job(f.n_clusters, cid, r);
    if (jr >= f.J) return false;
    const int rank = (int)jr / f.a.H;
    I.h = (int)jr - rank * f.a.H;
    I.n = f.ordered ? (int)f.order[rank] : rank;
    if (f.a.cu_seqlens) {
        I.tok_begin = f.a.cu_seqlens[I.n];
        I.tok_end = f.a.cu_seqlens[I.n + 1];
    } else {
        I.tok_begin = (int64_t)I.n * f.a.seq_len;
        I.tok_end = I.tok_begin + f.a.seq_len;
    }
    I.nch = (int)((I.tok_end - I.tok_begin + kC - 1) / kC);
    return true;
}
// The one job of a chain CTA of the two-kernel schedule: the chunks that the pass has of its (sequence, head), or a
// segment of them.
template <int kSeg>
__device__ __forceinline__ bool pass_job(const FusedArgs& f, int id, int r, JobInfo& I) {
    if (r > 0) return false;
    const ChunkArgs& a = f.a;
    const SegInfo s = seg_info<kSeg>(f, id);
    id = s.chain;
    const int rank = id / a.H;
    I.n = f.ordered ? (int)f.order[rank] : f.n_begin + rank;
    I.h = id - rank * a.H;
    int64_t cb, ce, tok0;
    if (a.cu_seqlens) {
        cb = a.chunk_cu[I.n]; ce = a.chunk_cu[I.n + 1];
        tok0 = a.cu_seqlens[I.n]; I.tok_end = a.cu_seqlens[I.n + 1];
    } else {
        cb = (int64_t)I.n * a.chunks_per_seq; ce = cb + a.chunks_per_seq;
        tok0 = (int64_t)I.n * a.seq_len; I.tok_end = tok0 + a.seq_len;
    }
    const int64_t first = cb < a.g0 ? a.g0 : cb;
    if (ce > a.g1) ce = a.g1;
    I.nch = ce > first ? (int)(ce - first) : 0;
    I.tok_begin = tok0 + (first - cb) * kC;
    I.tile0 = (first - a.g0) * a.H + I.h;
    if (kSeg) {
        const int len = (I.nch + f.seg_P - 1) / f.seg_P;
        const int c0 = s.p * len < I.nch ? s.p * len : I.nch, c1 = c0 + len < I.nch ? c0 + len : I.nch;
        I.nch = c1 - c0;
        I.tok_begin += (int64_t)c0 * kC;
        I.tile0 += (int64_t)c0 * a.H;
    }
    return true;
}
__device__ __forceinline__ bool call_aborted(const FusedArgs& f) {
    return *reinterpret_cast<volatile unsigned int*>(&f.hdr->abort_epoch) == f.epoch;
}
__device__ __forceinline__ void report(const FusedArgs& f, kda_status_t code, int where) {
    if (atomicCAS(&f.hdr->status, 0, (int)code) == 0) f.hdr->where = where;
    *reinterpret_cast<volatile unsigned int*>(&f.hdr->abort_epoch) = f.epoch;
    __threadfence();
}

// One (chunk, head) tile as the engine's service thread hands it to the other 255 threads.
struct TileDesc {
    long long tok0;                  // first token of the chunk
    char* tile;                      // where it goes
    int h;
    int len;                         // valid tokens, 1..64; 0 = no more tiles for this engine
    int pad[10];
};
static_assert(sizeof(TileDesc) == 64, "three descriptors fit the 192 bytes reserved");

// The tiles of a cluster are numbered through its jobs; engine e of E makes tiles e, e + E, ..., its m-th
// tile in position m % depth of its own share of the cluster's ring.
struct EngineCursor {
    int cid, e;
    int r, c, m;                     // job, chunk inside it, tiles handed out so far
    uint32_t ready;                  // shared::cluster address of the chain's barriers of this engine's positions
    int done, published;             // tiles finished, and announced to the chain
};
static_assert(sizeof(EngineCursor) <= 64, "fits the 64 bytes reserved");
__device__ void cluster_tile(const FusedArgs& f, EngineCursor& k, TileDesc* d)
{
    d->len = 0;
    JobInfo J;
    for (;;) {
        if (!job_info(f, k.cid, k.r, J)) return;
        if (k.c < J.nch) break;
        k.c -= J.nch;
        ++k.r;
    }
    d->tok0 = J.tok_begin + (int64_t)k.c * kC;
    const int64_t rem = J.tok_end - d->tok0;
    d->tile = f.ring + (size_t)((k.cid * f.n_eng + k.e) * f.depth + k.m % f.depth) * tc::TILE_BYTES;
    d->h = J.h;
    d->len = rem < kC ? (int)rem : kC;
    k.c += f.n_eng;
    ++k.m;
}

// ====================================================================================================
// intra-chunk engine: 256 threads (te = 0..255), named barrier `bar_id`, 256 TMEM columns at tmem_e
// ====================================================================================================
// Stand-alone use (kFused = false, the intra-chunk kernel of the two-kernel schedule): tile number
// idx of the pass = (chunk of the pass) * H + head goes to position idx of a plain tile array, the
// engines take the tiles first, first + stride, ...; nothing is waited for or published.
__device__ bool static_tile(const FusedArgs& f, uint32_t idx, TileDesc* d)
{
    d->len = 0;
    if (idx >= f.n_prod) return false;
    const uint32_t gl = idx / (uint32_t)f.a.H;
    const ChunkLoc L = locate_chunk(f.a, f.a.g0 + gl);
    d->tok0 = L.tok0;
    d->tile = f.ring + (size_t)idx * tc::TILE_BYTES;
    d->h = (int)(idx - gl * (uint32_t)f.a.H);
    d->len = L.len;
    return true;
}

template <bool kHasQ, bool kFused, bool kLayer = false>
__device__ void engine_run(const FusedArgs& f, uint8_t* smem, uint32_t tmem_e, int bar_id, int te,
                           uint32_t first, uint32_t stride, const CUtensorMap* tm_k,
                           const CUtensorMap* tm_q, const CUtensorMap* tm_v)
{
    constexpr bool has_q = kHasQ;
    // rows of the gating loop at once: the fewer, the less code.  4096 x 32 heads, fused, 8 / 4 / 2: 113.6, 113.0, 115.1 us; 128 Ki tokens
    // for the state, fused: 2800, 2743, 2567 (one row: 2886); layer call on three prompts: 218.4, 222.8, 223.9
    constexpr int kNW = 8, kRPT = 8, kGateRows = kLayer ? 8 : kFused && !kHasQ ? 2 : 4;
    constexpr int kInvWarps = 6;       // warps of the blocked substitution
    constexpr int kMma2Warp = 2;       // issues half of the second MMA group (warp 0 the rest)
    const ChunkArgs& a = f.a;
    float* sA = reinterpret_cast<float*>(smem + E_A);
    float* sTd = reinterpret_cast<float*>(smem + E_TD);
    float* sTot = reinterpret_cast<float*>(smem + E_TD);   // [8][128] during the scan
    float* sBeta = reinterpret_cast<float*>(smem + E_BETA);
    TileDesc* desc = reinterpret_cast<TileDesc*>(smem + E_DESC);
    uint64_t* mma_bar = reinterpret_cast<uint64_t*>(smem + E_BAR);
    uint64_t* bar_k = mma_bar + 1;   // raw k has landed in the staging buffer
    uint64_t* bar_q = mma_bar + 3;   // raw q has landed in rows 64-127 of the operand image
    uint64_t* bar_v = mma_bar + 5;   // v has landed
    uint64_t* bar_free = mma_bar + 6;   // [depth] (kFused) the chain has read a ring position
    volatile uint32_t* abort_word = reinterpret_cast<volatile uint32_t*>(mma_bar + 2);

    const int warp = ptx::warp_uniform(te >> 5), lane = te & 31;
    auto ebar = [&]() { ptx::named_bar_sync(bar_id, kEngThreads); };
    auto inv_bar = [&]() { ptx::named_bar_sync(bar_id + 2, kInvWarps * 32); };

    // thread (w, c4) owns rows 8w..8w+7 and channels 4c4..4c4+3 in the gating phase
    const int c4 = lane, d0 = c4 * 4, i0 = warp * kRPT;
    float G[kRPT][4];
    float rate = 0.f, bias[4] = {0.f, 0.f, 0.f, 0.f};   // layer mode: decay-function parameters of the tile's head
    auto prefetch_regs = [&](const TileDesc& D) {
        if (kLayer) {
            // bf16 pre-activations of the decay function; the function itself is applied at the top of
            // the tile, when the registers are next looked at
            const __nv_bfloat16* gp = reinterpret_cast<const __nv_bfloat16*>(a.log_alpha) +
                                      ((size_t)D.tok0 * a.H + D.h) * kD + d0;
#pragma unroll
            for (int r = 0; r < kRPT; ++r) {
                const int i = i0 + r;
                uint32_t lo = 0u, hi = 0u;
                if (i < D.len)
                    asm volatile("ld.global.L1::no_allocate.v2.u32 {%0,%1}, [%2];"
                                 : "=r"(lo), "=r"(hi)
                                 : "l"(gp + (size_t)i * a.H * kD));
                G[r][0] = __uint_as_float(lo);    // (unpacked when they are used: nothing here waits for the loads)
                G[r][1] = __uint_as_float(hi);
            }
            rate = a.gate_rate[D.h];
            const float4 b4 = *reinterpret_cast<const float4*>(a.gate_bias + (size_t)D.h * kD + d0);
            bias[0] = b4.x; bias[1] = b4.y; bias[2] = b4.z; bias[3] = b4.w;
            return;
        }
        const float* gp = a.log_alpha + ((size_t)D.tok0 * a.H + D.h) * kD + d0;
#pragma unroll
        for (int r = 0; r < kRPT; ++r) {
            const int i = i0 + r;
            if (i < D.len) {
                ld_f4(gp + (size_t)i * a.H * kD, G[r][0], G[r][1], G[r][2], G[r][3]);
            } else {
                G[r][0] = G[r][1] = G[r][2] = G[r][3] = 0.f;
            }
        }
    };
    // k, q, v of the NEXT tile by 2-D tiled TMA loads (128-byte swizzle), each requested as soon as
    // its destination is free: k into a staging buffer (the gating loop reads it there and writes
    // the gated image), q straight into rows 64-127 of the operand image (gated in place), v into
    // the B operand buffer of the second MMA group; beta by small asynchronous copies.  Run by the
    // bulk thread (beta: by the first 64 threads).
    auto request_k = [&](const TileDesc& D) {
        ptx::mbar_expect_tx(bar_k, 16384);
#pragma unroll
        for (int hf = 0; hf < 2; ++hf)
            ptx::tma_load_2d(smem + E_KS + hf * 8192, tm_k, D.h * kD + hf * 64, (int)D.tok0, bar_k);
    };
    auto request_q = [&](const TileDesc& D) {
        ptx::mbar_expect_tx(bar_q, 16384);
#pragma unroll
        for (int hf = 0; hf < 2; ++hf)
            ptx::tma_load_2d(smem + E_KQ + hf * E_KQ_HALF + 8192, tm_q, D.h * kD + hf * 64, (int)D.tok0, bar_q);
    };
    auto request_v = [&](const TileDesc& D) {
        ptx::mbar_expect_tx(bar_v, 16384);
#pragma unroll
        for (int hf = 0; hf < 2; ++hf)
            ptx::tma_load_2d(smem + E_V + hf * E_V_BLOCK, tm_v, D.h * kD + hf * 64, (int)D.tok0, bar_v);
    };
    auto request_beta = [&](const TileDesc& D) {
        if (te < kC) {
            const bool ok = te < D.len;
            ptx::cp_async4(sBeta + te, a.beta + (D.tok0 + (ok ? te : 0)) * a.H + D.h, ok ? 4u : 0u);
        }
        ptx::cp_async_commit();
    };

    bool timed_out = false, out_of_range = false;
    bool pend_k = false, pend_q = false, pend_v = false;   // (thread 0) requests not yet waited for
    uint32_t tma_parity = 0;
    uint32_t next_static = first;
    int cur = 0;
    EngineCursor& cursor = *reinterpret_cast<EngineCursor*>(smem + E_CUR);   // (service thread, kFused)
    auto publish = [&]() {   // (the tile's stores are performed)
        if (cursor.published == cursor.done) return;
        ptx::mbar_arrive_cluster(cursor.ready + (uint32_t)(cursor.published % f.depth) * 8u);
        ++cursor.published;
    };
    bool staged = false;             // W and U^T of the tile before this one lie in their staging buffers
    auto store_staged = [&](char* to) {   // (service thread)
        ptx::bulk_s2g(to + tc::OFF_QW, smem + E_V, 8192);
        ptx::bulk_s2g(to + tc::OFF_QW + tc::QW_HALF, smem + E_V + 8192, 8192);
        ptx::bulk_s2g(to + tc::OFF_U, smem + E_A, 16384);
        ptx::bulk_commit();
        if (kFused) ++cursor.done;
    };
    auto find_tile = [&](TileDesc* d) {   // (service thread)
        if (kFused) {
            cluster_tile(f, cursor, d);
        } else {
            static_tile(f, next_static, d);
            next_static += stride;
        }
    };
    if (te == kServiceThread) {
        find_tile(&desc[0]);
        if (desc[0].len > 0) find_tile(&desc[1]);
        else desc[1].len = 0;
    }
    ebar();
    if (desc[0].len > 0 && !*abort_word) {
        prefetch_regs(desc[0]);
        if (te == kServiceThread) {
            request_k(desc[0]);
            if (has_q) request_q(desc[0]);
        }
        request_beta(desc[0]);
        pend_k = true;
        pend_q = has_q;
    }
    KT_DECL(10);
    while (true) {
        // (the descriptors are read where they are used: registers are short)
        const TileDesc& D = desc[cur];
        const int d_len = D.len;
        if (d_len == 0) break;       // (an abort is looked at behind a barrier only)
        KT_MARK(te == 0, 0);   // loop overhead

        if (kLayer) {
            // log2 alpha = -exp(rate) * log2(1 + e^(x + bias)); rows past the end of the sequence do not decay
            const float nr = -__expf(rate);
            float b2[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) b2[e] = bias[e] * kLog2e;
#pragma unroll
            for (int r = 0; r < kRPT; ++r) {
                const uint32_t lo = __float_as_uint(G[r][0]), hi = __float_as_uint(G[r][1]);
                const float x[4] = {__uint_as_float(lo << 16), __uint_as_float(lo & 0xffff0000u), __uint_as_float(hi << 16),
                                    __uint_as_float(hi & 0xffff0000u)};
                const float nrr = i0 + r < d_len ? nr : 0.f;
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float x2 = fmaf(x[e], kLog2e, b2[e]);
                    G[r][e] = fmaf(nrr, fmaxf(x2, 0.f) + lg2(1.f + ex2(-fabsf(x2))), r > 0 ? G[r - 1][e] : 0.f);
                }
            }
        }
        // ---- a1: cumulative log-decay, in the log2 domain (exponentials below are bare ex2) ---------
        if (!kLayer) {
#pragma unroll
            for (int e = 0; e < 4; e += 2) set(&G[0][e], __fmul2_rn(pair(&G[0][e]), both(kLog2e)));
#pragma unroll
            for (int r = 1; r < kRPT; ++r)
#pragma unroll
                for (int e = 0; e < 4; e += 2) set(&G[r][e], __ffma2_rn(pair(&G[r][e]), both(kLog2e), pair(&G[r - 1][e])));
        }
        *reinterpret_cast<float4*>(sTot + warp * kD + d0) =
            make_float4(G[kRPT - 1][0], G[kRPT - 1][1], G[kRPT - 1][2], G[kRPT - 1][3]);
        ptx::cp_async_wait_all();             // beta
        if (kLayer && te < kC)                // (each of these threads copied its own element)
            sBeta[te] = te < d_len ? 1.f / (1.f + __expf(-sBeta[te])) : 0.f;
        ebar();
        KT_MARK(te == 0, 1);   // scan
        if (te == kServiceThread && staged) store_staged(desc[cur == 0 ? 2 : cur - 1].tile);
        staged = false;
        if (*abort_word) break;
        float base[4] = {0.f, 0.f, 0.f, 0.f}, gref[4], glast[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int r2 = 0; r2 < kNW; ++r2) {
            const float4 x4 = *reinterpret_cast<const float4*>(sTot + r2 * kD + d0);
            const float x[4] = {x4.x, x4.y, x4.z, x4.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                if (r2 < warp) base[e] += x[e];
                glast[e] += x[e];
            }
        }
        // reference of the decay factorisation: half the chunk's total log-decay, per channel, so that
        // |G_i - G_ref| <= |G_C| / 2 (+ 1/2) for every row whatever the distribution of the decay over the chunk
#pragma unroll
        for (int e = 0; e < 4; ++e) gref[e] = (0.5f * glast[e] + 12582912.f) - 12582912.f;   // to a whole number
        float em[4];   // exp(G_m), a power of two
#pragma unroll
        for (int e = 0; e < 4; ++e) em[e] = ex2(gref[e]);
        if (warp == 0) {
            float ec[4];   // exp(G_C - G_m)
#pragma unroll
            for (int e = 0; e < 4; ++e) ec[e] = ex2(glast[e] - gref[e]);
            *reinterpret_cast<float4*>(smem + E_GV + d0 * 4) =
                make_float4(ec[0] * em[0], ec[1] * em[1], ec[2] * em[2], ec[3] * em[3]);
            *reinterpret_cast<float4*>(smem + E_GV + 512 + d0 * 4) = make_float4(ec[0], ec[1], ec[2], ec[3]);
            *reinterpret_cast<float4*>(smem + E_EM + d0 * 4) = make_float4(em[0], em[1], em[2], em[3]);
            // a channel that decays by more than e^-160 inside this chunk leaves the range of the
            // two-factor form: flag it (the clamp below keeps everything finite)
            if (fminf(fminf(glast[0], glast[1]), fminf(glast[2], glast[3])) < -2.f * kClamp2) out_of_range = true;
        }
#ifdef KDA_FUSED_TIMING
        if (te == 0) {
            const uint64_t now_ = ptx::globaltimer_ns();
        }
#endif
        if (!ptx::mbar_wait(bar_k, tma_parity, f.a.wait_limit_ns)) timed_out = true;   // raw k, q have landed
        if (has_q && !ptx::mbar_wait(bar_q, tma_parity, f.a.wait_limit_ns)) timed_out = true;
        pend_k = pend_q = false;
        KT_MARK(te == 0, 2);   // prefix + TMA wait
        // ---- gated operands ---------------------------------------------------------------------------
        // (the clamp is for channels that reach it, see out_of_range; a second copy of the loop without it, chosen per warp,
        // cost more in fetched instructions than it saved: packed batch, two kernels, 3053 instead of 2944 us.  Rolled for the
        // same reason.)
        float* sNorm = reinterpret_cast<float*>(smem + E_NORM);
        if (kLayer) {
            // L2Norm of k and q: the warp owns its eight rows whole (32 lanes x 4 channels)
            const int hf = c4 >> 4;
            float ss[2 * kRPT];   // k rows, q rows
#pragma unroll
            for (int r = 0; r < kRPT; ++r) {
                const int i = i0 + r;
                const uint32_t o2 = (uint32_t)(i * 128 + ((((c4 >> 1) & 7) ^ (i & 7)) << 4) + (c4 & 1) * 8);
                const uint2 k2 = *reinterpret_cast<const uint2*>(smem + E_KS + hf * 8192 + o2);
                uint2 q2 = make_uint2(0u, 0u);
                if (has_q) q2 = *reinterpret_cast<const uint2*>(smem + E_KQ + hf * E_KQ_HALF + o2 + 8192);
                const float k0 = __uint_as_float(k2.x << 16), k1 = __uint_as_float(k2.x & 0xffff0000u);
                const float k2f = __uint_as_float(k2.y << 16), k3 = __uint_as_float(k2.y & 0xffff0000u);
                const float q0 = __uint_as_float(q2.x << 16), q1 = __uint_as_float(q2.x & 0xffff0000u);
                const float q2f = __uint_as_float(q2.y << 16), q3 = __uint_as_float(q2.y & 0xffff0000u);
                ss[r] = k0 * k0 + k1 * k1 + k2f * k2f + k3 * k3;
                ss[kRPT + r] = q0 * q0 + q1 * q1 + q2f * q2f + q3 * q3;
            }
            // sums over the 32 lanes: each exchange halves the values a lane still carries (16 shuffles, not 80)
#pragma unroll
            for (int n = kRPT, x = 16; n >= 1; n >>= 1, x >>= 1) {
                const bool up = (lane & x) != 0;
#pragma unroll
                for (int i = 0; i < n; ++i) {
                    const float send = up ? ss[i] : ss[i + n], keep = up ? ss[i + n] : ss[i];
                    ss[i] = keep + __shfl_xor_sync(0xffffffffu, send, x);
                }
            }
            ss[0] += __shfl_xor_sync(0xffffffffu, ss[0], 1);
            if ((lane & 1) == 0) {   // (rows past the end of the sequence are zeroed below: finite factor)
                const int v = lane >> 1, r = v & (kRPT - 1);
                sNorm[(v >= kRPT ? kC : 0) + i0 + r] = i0 + r < d_len ? rsqrtf(ss[0] + a.l2_eps) : 0.f;
            }
            __syncwarp();
        }
        {
            const int hf = c4 >> 4;                       // K-half (channels 0-63 / 64-127)
            float off[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) off[e] = base[e] - gref[e];
#pragma unroll 1
            for (int r0 = 0; r0 < kRPT; r0 += kGateRows) {
#pragma unroll
                for (int r = 0; r < kGateRows; ++r) {
                    const int i = i0 + r0 + r;
                    const uint32_t o2 = (uint32_t)(i * 128 + ((((c4 >> 1) & 7) ^ (i & 7)) << 4) + (c4 & 1) * 8);
                    uint8_t* pk = smem + E_KQ + hf * E_KQ_HALF + o2;
                    uint2 k2 = *reinterpret_cast<const uint2*>(smem + E_KS + hf * 8192 + o2);
                    uint2 q2 = make_uint2(0u, 0u);
                    if (has_q) q2 = *reinterpret_cast<const uint2*>(pk + 8192);
                    if (i >= d_len) k2 = q2 = make_uint2(0u, 0u);
                    const float kf[4] = {__uint_as_float(k2.x << 16), __uint_as_float(k2.x & 0xffff0000u),
                                         __uint_as_float(k2.y << 16), __uint_as_float(k2.y & 0xffff0000u)};
                    const float qf[4] = {__uint_as_float(q2.x << 16), __uint_as_float(q2.x & 0xffff0000u),
                                         __uint_as_float(q2.y << 16), __uint_as_float(q2.y & 0xffff0000u)};
                    float okg[4], oqg[4], oki[4];
                    float rk = 1.f, rq = a.scale;
                    if (kLayer) {
                        rk = sNorm[i];
                        rq = a.scale * sNorm[kC + i];
                    }
#pragma unroll
                    for (int e = 0; e < 4; e += 2) {
                        const float2 x2 = __fadd2_rn(pair(&G[r][e]), pair(&off[e]));
                        const float x0 = fminf(fmaxf(x2.x, -kClampX), kClampX), x1 = fminf(fmaxf(x2.y, -kClampX), kClampX);
                        float2 e1 = make_float2(ex2(x0), ex2(x1)), e2 = make_float2(ex2(-x0), ex2(-x1));   // exp(G - G_m), exp(G_m - G)
                        set(&oqg[e], __fmul2_rn(__fmul2_rn(both(rq), pair(&qf[e])), e1));
                        if (kLayer) {
                            e1 = __fmul2_rn(e1, both(rk));
                            e2 = __fmul2_rn(e2, both(rk));
                        }
                        set(&okg[e], __fmul2_rn(pair(&kf[e]), e1));
                        set(&oki[e], __fmul2_rn(pair(&kf[e]), e2));
                    }
                    *reinterpret_cast<uint2*>(pk) = make_uint2(pack_bf16(okg[0], okg[1]), pack_bf16(okg[2], okg[3]));
                    if (has_q)
                        *reinterpret_cast<uint2*>(pk + 8192) =
                            make_uint2(pack_bf16(oqg[0], oqg[1]), pack_bf16(oqg[2], oqg[3]));
                    *reinterpret_cast<uint2*>(smem + E_KI + hf * E_KI_HALF + o2) =
                        make_uint2(pack_bf16(oki[0], oki[1]), pack_bf16(oki[2], oki[3]));
                    if (has_q)   // what the chain reads: scale Q exp(G), over the raw k that this thread has just read
                        *reinterpret_cast<uint2*>(smem + E_KS + hf * 8192 + o2) =
                            make_uint2(pack_bf16(__fmul2_rn(pair(oqg), pair(em))), pack_bf16(__fmul2_rn(pair(oqg + 2), pair(em + 2))));
                }
#pragma unroll
                for (int r = 0; r + kGateRows < kRPT; ++r)
#pragma unroll
                    for (int e = 0; e < 4; ++e) G[r][e] = G[r + kGateRows][e];
            }
        }
        if (te == kServiceThread) ptx::bulk_wait_read0();   // the previous tile's W and U^T have been read out
        ptx::fence_async_smem();
        ptx::tc_fence_before();
        ebar();
        ptx::tc_fence_after();
        KT_MARK(te == 0, 3);   // gating

        // ---- a2 + a5: [Kg ; Qg] Ki^T --------------------------------------------------------------------
        if (te == kServiceThread) {
            if (kFused) {
                if (f.depth == 1) {      // (the chain needs the previous tile to give its position back)
                    ptx::bulk_wait_all0();
                    publish();
                }
                const int m = cursor.done;
                if (m >= f.depth) {
                    const uint64_t t0 = ptx::globaltimer_ns();
                    while (!ptx::mbar_try_cluster(&bar_free[m % f.depth], (uint32_t)(m / f.depth - 1) & 1u)) {
                        if (*abort_word || call_aborted(f)) { *abort_word = 1; break; }
                        if (ptx::globaltimer_ns() - t0 > f.a.wait_limit_ns) { timed_out = true; *abort_word = 1; break; }
                    }
                    ptx::fence_async_global();
                }
            }
            if (has_q) {
                ptx::bulk_s2g(D.tile + tc::OFF_QW + 8192, smem + E_KS, 8192);
                ptx::bulk_s2g(D.tile + tc::OFF_QW + tc::QW_HALF + 8192, smem + E_KS + 8192, 8192);
            }
            ptx::bulk_s2g(D.tile + tc::OFF_KI, smem + E_KI, 16384);
            ptx::bulk_s2g(D.tile + tc::OFF_GV, smem + E_GV, tc::GV_BYTES);
            ptx::bulk_commit();
            request_v(D);            // over W
        }
        pend_v = true;
        if (warp == 0) {
            const uint32_t idesc = ptx::umma_idesc_bf16(128, 64);
            const uint32_t a0 = ptx::smem_u32(smem + E_KQ), b0 = ptx::smem_u32(smem + E_KI);
#pragma unroll
            for (int k = 0; k < 8; ++k)
                ptx::umma_bf16(tmem_e, ptx::umma_desc_sw128(a0 + (k >> 2) * E_KQ_HALF + (k & 3) * 32),
                               ptx::umma_desc_sw128(b0 + (k >> 2) * E_KI_HALF + (k & 3) * 32), idesc, k > 0);
            ptx::umma_commit(mma_bar);
        }
        if (warp == kMma2Warp) ptx::umma_commit(mma_bar);   // (the barrier counts both issuing warps)
        const int nxt = cur == 2 ? 0 : cur + 1, nxt2 = nxt == 2 ? 0 : nxt + 1;
        const TileDesc& Dn = desc[nxt];
        const bool has_next = Dn.len > 0 && !*abort_word;
        if (has_next) {
            prefetch_regs(Dn);   // the next tile's log alpha: its registers are free since the gating loop
            pend_k = true;
        }
        if (!ptx::mbar_wait(mma_bar, 0, f.a.wait_limit_ns)) timed_out = true;
        ptx::tc_fence_after();
        KT_MARK(te == 0, 4);   // MMA A
        {
            const int q4 = warp & 3, c0 = (warp >> 2) * 32;
            const int Rr = q4 * 32 + lane;
            uint32_t r[32];
            // the warp's block of 32 rows lies above the diagonal, below it, or on it: only the last needs masks, the first is
            // zero (and of L nobody reads it)
            const int where = (q4 & 1) * 32 - c0;      // > 0: below
            if (where >= 0) {
                ptx::tmem_ld_32x32b_x32(tmem_e + ((uint32_t)(q4 * 32) << 16) + c0, r);
                ptx::tmem_ld_wait();
            }
            if (Rr < 64) {
                const int i = Rr, lim = where > 0 ? 32 : lane;
                const float bi = sBeta[i];
                if (where >= 0) {
#pragma unroll
                    for (int j4 = 0; j4 < 32; j4 += 4) {
                        float x[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) x[e] = j4 + e < lim ? bi * __uint_as_float(r[j4 + e]) : 0.f;
                        *reinterpret_cast<float4*>(sA + i * LDT + c0 + j4) = make_float4(x[0], x[1], x[2], x[3]);
                    }
                }
            } else if (has_q) {
                const int i = Rr - 64, lim = where > 0 ? 32 : where < 0 ? -1 : lane;
#pragma unroll
                for (int j8 = 0; j8 < 32; j8 += 8) {
                    float x[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) x[e] = j8 + e <= lim ? __uint_as_float(r[j8 + e]) : 0.f;
                    *reinterpret_cast<uint4*>(smem + E_AQ + ptx::sw128_off(i, c0 + j8)) =
                        make_uint4(pack_bf16(x[0], x[1]), pack_bf16(x[2], x[3]), pack_bf16(x[4], x[5]),
                                   pack_bf16(x[6], x[7]));
                }
            }
        }
        ptx::fence_async_smem();
        ptx::tc_fence_before();
        ebar();
        if (te == kServiceThread) {
            if (has_q) {
                ptx::bulk_s2g(D.tile + tc::OFF_AQ, smem + E_AQ, 8192);
                ptx::bulk_commit();
            }
            ptx::bulk_wait_read0();   // Q, K' and Aqk have been read out: the next q and k may land over them
            if (has_next) {
                request_k(Dn);
                if (has_q) request_q(Dn);
            }
            if (has_next) find_tile(&desc[nxt2]);
            else desc[nxt2].len = 0;
            if (kFused && f.depth > 1) {   // the previous tile (its stores are older than this tile's): the arrival takes a while
                ptx::bulk_wait_all<has_q ? 2 : 1>();
                publish();
            }
        }
        KT_MARK(te == 0, 5);   // A read-out

        // ---- a3: T = (I + L)^-1, blocked forward substitution -------------------------------------------
        // T's diagonal blocks live in sTd, its sub-diagonal block (I, J) in the (J, I) position of sA
        // (the upper triangle of L is empty), so L, X and T share one 64 x 64 array.
        auto blkA = [&](int I, int J) { return sA + (I * 16) * LDT + J * 16; };
        auto blkD = [&](int I) { return sTd + I * 16 * LDD; };
        if (te < 64) {   // diagonal 16x16 blocks: one column per thread, rows unrolled in registers
            const int I = te >> 4, c = te & 15;
            const float* Lb = blkA(I, I);
            float x[16];
#pragma unroll
            for (int r = 0; r < 16; ++r) {
                float s = (r == c) ? 1.f : 0.f;
#pragma unroll
                for (int m4 = 0; m4 < r; m4 += 4) {
                    const float4 l4 = *reinterpret_cast<const float4*>(Lb + r * LDT + m4);
                    const float l[4] = {l4.x, l4.y, l4.z, l4.w};
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (m4 + e < r) s -= l[e] * x[m4 + e];
                }
                x[r] = s;
            }
#pragma unroll
            for (int r = 0; r < 16; ++r) blkD(I)[r * LDD + c] = x[r];
        }
        if (warp < kInvWarps) inv_bar();
        // X_IM = T_II L_IM for the six sub-diagonal blocks (one warp each, in place), then
        // T_IJ = - sum_{M=J..I-1} X_IM T_MJ in three dependency stages; the terms of a sum that do not
        // depend on blocks still being computed are taken early (kept, un-negated, in the block's place).
        //   stage A: T10, T21, T32 final;  P20 = X20 T00,  P31 = X31 T11,  P30 = X30 T00
        //   stage B: T20 = -(P20 + X21 T10),  T31 = -(P31 + X32 T21),  P30 += X31 T10
        //   stage C: T30 = -(P30 + X32 T20)
        if (warp < 6) {
            const int I = warp < 1 ? 1 : (warp < 3 ? 2 : 3);
            const int M = warp < 1 ? 0 : (warp < 3 ? warp - 1 : warp - 3);
            float acc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
            block16_mma(acc, blkD(I), LDD, blkA(I, M), LDT, lane);
            __syncwarp();   // every lane has read its part of L_IM before anyone overwrites it
            block16_store(blkA(I, M), acc, 1.f, LDT, lane);
            __syncwarp();
            float acc2[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
            block16_mma(acc2, blkA(I, M), LDT, blkD(M), LDD, lane);
            block16_store(blkA(M, I), acc2, (I - M == 1) ? -1.f : 1.f, LDT, lane);
        }
        if (warp < kInvWarps) inv_bar();
        if (warp < 3) {
            // warp 0: T20 (M = 1), warp 1: T31 (M = 2), warp 2: P30 += X31 T10
            const int I = warp == 0 ? 2 : 3, J = warp == 1 ? 1 : 0, M = warp == 1 ? 2 : 1;
            float acc[2][4];
            block16_load(acc, blkA(J, I), LDT, lane);
            block16_mma(acc, blkA(I, M), LDT, blkA(J, M), LDT, lane);
            block16_store(blkA(J, I), acc, warp < 2 ? -1.f : 1.f, LDT, lane);
        }
        if (warp < kInvWarps) inv_bar();
        if (warp == 0) {
            float acc[2][4];
            block16_load(acc, blkA(0, 3), LDT, lane);
            block16_mma(acc, blkA(3, 2), LDT, blkA(0, 2), LDT, lane);
            block16_store(blkA(0, 3), acc, -1.f, LDT, lane);
        }
        if (has_next) pend_q = has_q;
        if (!ptx::mbar_wait(bar_v, tma_parity, f.a.wait_limit_ns)) timed_out = true;   // v has landed
        pend_v = false;
        tma_parity ^= 1;
        if (d_len < kC) {   // short last chunk: rows past the end hold other tokens' v; zero them
            for (int idx = te; idx < (kC - d_len) * 16; idx += kEngThreads) {
                const int j = d_len + (idx >> 4), c16 = idx & 15;
                *reinterpret_cast<uint4*>(smem + E_V + (c16 >> 3) * E_V_BLOCK + j * 128 +
                                          (((c16 & 7) ^ (j & 7)) << 4)) = make_uint4(0u, 0u, 0u, 0u);
            }
        }
        ebar();
        KT_MARK(te == 0, 6);   // inverse

        // ---- a4: Mm = T Diag(beta) as the A operand; [W | U] = Mm [Kg | V] ---------------------------------
        {
            const int i = te & 63, J = te >> 6, I = i >> 4;   // one 16-column block of one row per thread
            const int j0 = J * 16;
            float x[16];
            if (J > I) {
#pragma unroll
                for (int e = 0; e < 16; ++e) x[e] = 0.f;
            } else {
                const float* src = (J == I) ? blkD(I) + (i & 15) * LDD : blkA(J, I) + (i & 15) * LDT;
#pragma unroll
                for (int e4 = 0; e4 < 16; e4 += 4) {
                    const float4 tv = *reinterpret_cast<const float4*>(src + e4);
                    const float4 bv = *reinterpret_cast<const float4*>(sBeta + j0 + e4);
                    set(x + e4, __fmul2_rn(make_float2(tv.x, tv.y), make_float2(bv.x, bv.y)));
                    set(x + e4 + 2, __fmul2_rn(make_float2(tv.z, tv.w), make_float2(bv.z, bv.w)));
                }
            }
#pragma unroll
            for (int c8 = 0; c8 < 2; ++c8) {
                const uint4 pk = make_uint4(pack_bf16(x[c8 * 8], x[c8 * 8 + 1]), pack_bf16(x[c8 * 8 + 2], x[c8 * 8 + 3]),
                                            pack_bf16(x[c8 * 8 + 4], x[c8 * 8 + 5]), pack_bf16(x[c8 * 8 + 6], x[c8 * 8 + 7]));
                uint8_t* dst = smem + E_KI + i * 128 + ((((j0 >> 3) + c8) ^ (i & 7)) << 4);
                *reinterpret_cast<uint4*>(dst) = pk;
                *reinterpret_cast<uint4*>(dst + 8192) = pk;   // rows 64-127 repeat rows 0-63
            }
        }
        ptx::fence_async_smem();
        ptx::tc_fence_before();
        ebar();
        if (warp == 0) {
            ptx::tc_fence_after();
            const uint32_t idesc = ptx::umma_idesc_bf16(128, 128) | ptx::kIdescBMajorMN;
            const uint32_t m0 = ptx::smem_u32(smem + E_KI);
            const uint32_t kg0 = ptx::smem_u32(smem + E_KQ);
#pragma unroll
            for (int k = 0; k < 4; ++k)
                ptx::umma_bf16(tmem_e, ptx::umma_desc_sw128(m0 + k * 32),
                               ptx::umma_desc_sw128_mn(kg0 + k * 2048, E_KQ_HALF), idesc, k > 0);
            ptx::umma_commit(mma_bar);
        }
        if (warp == kMma2Warp) {   // U^T = V^T Mm^T (the chain has its columns in the TMEM lanes), issued at the same time
            ptx::tc_fence_after();
            const uint32_t m0 = ptx::smem_u32(smem + E_KI), v0 = ptx::smem_u32(smem + E_V);
#pragma unroll
            for (int k = 0; k < 4; ++k)
                ptx::umma_bf16(tmem_e + 128, ptx::umma_desc_sw128_mn(v0 + k * 2048, E_V_BLOCK), ptx::umma_desc_sw128(m0 + k * 32),
                               ptx::umma_idesc_bf16(128, 64) | ptx::kIdescAMajorMN, k > 0);
            ptx::umma_commit(mma_bar);
        }
        if (!ptx::mbar_wait(mma_bar, 1, f.a.wait_limit_ns)) timed_out = true;
        KT_MARK(te == 0, 7);   // Mm + MMA B
        if (has_next) request_beta(Dn);   // (beta is free)
        ptx::tc_fence_after();
        {   // W' rows lie in TMEM lanes 0-63 and again in 64-127: 32 columns a warp; U^T has a lane per column of U
            const int q4 = warp & 3, g = warp >> 2, i = (q4 & 1) * 32 + lane;
            const uint32_t tq = tmem_e + ((uint32_t)(q4 * 32) << 16);
            const int col0 = (g * 2 + (q4 >> 1)) * 32;
            uint32_t r[32];
            ptx::tmem_ld_32x32b_x32(tq + col0, r);
            ptx::tmem_ld_wait();
#pragma unroll
            for (int j8 = 0; j8 < 32; j8 += 8) {   // W = exp(G_m) . W'
                const float4 e0 = *reinterpret_cast<const float4*>(smem + E_EM + (col0 + j8) * 4);
                const float4 e1 = *reinterpret_cast<const float4*>(smem + E_EM + (col0 + j8) * 4 + 16);
                *reinterpret_cast<uint4*>(smem + E_V + (col0 >> 6) * 8192 + ptx::sw128_off(i, (col0 & 63) + j8)) =
                    make_uint4(pack_bf16(__fmul2_rn(make_float2(__uint_as_float(r[j8]), __uint_as_float(r[j8 + 1])), make_float2(e0.x, e0.y))),
                               pack_bf16(__fmul2_rn(make_float2(__uint_as_float(r[j8 + 2]), __uint_as_float(r[j8 + 3])), make_float2(e0.z, e0.w))),
                               pack_bf16(__fmul2_rn(make_float2(__uint_as_float(r[j8 + 4]), __uint_as_float(r[j8 + 5])), make_float2(e1.x, e1.y))),
                               pack_bf16(__fmul2_rn(make_float2(__uint_as_float(r[j8 + 6]), __uint_as_float(r[j8 + 7])), make_float2(e1.z, e1.w))));
            }
            ptx::tmem_ld_32x32b_x32(tq + 128 + g * 32, r);
            ptx::tmem_ld_wait();
#pragma unroll
            for (int j8 = 0; j8 < 32; j8 += 8)
                *reinterpret_cast<uint4*>(smem + E_A + tc::ut_off(q4 * 32 + lane, g * 4 + (j8 >> 3))) =
                    make_uint4(pack_bf16(__uint_as_float(r[j8]), __uint_as_float(r[j8 + 1])),
                               pack_bf16(__uint_as_float(r[j8 + 2]), __uint_as_float(r[j8 + 3])),
                               pack_bf16(__uint_as_float(r[j8 + 4]), __uint_as_float(r[j8 + 5])),
                               pack_bf16(__uint_as_float(r[j8 + 6]), __uint_as_float(r[j8 + 7])));
        }
        ptx::fence_async_smem();
        ptx::tc_fence_before();
        if (timed_out) *abort_word = 1;
        staged = true;               // stored after the next barrier
        KT_MARK(te == 0, 8);   // epilogue
#ifdef KDA_FUSED_TIMING
        if (te == 0) kt_acc_[9] += 16;   // tiles
#endif
        cur = nxt;
    }   // tile loop
    KT_FLUSH(te == 0, f.hdr, 0, 10);

    ebar();
    if (te == kServiceThread && staged && !*abort_word) {
        const int last = cur == 0 ? 2 : cur - 1;
        store_staged(desc[last].tile);
    }
    if (timed_out) report(f, KDA_ERR_TIMEOUT, 10);
    if (out_of_range) atomicOr(&f.hdr->flags, 1);
    if (te == kServiceThread) {
        ptx::bulk_wait_all0();   // shared memory must outlive the reads of every bulk store
        if (kFused && !timed_out && !*abort_word) publish();
    }
    ptx::cp_async_wait_all();
    // an aborted engine may still have a TMA load in flight (requested for a tile it never started)
    if (te == 0) {
        // tma_parity is the parity of the current / next tile's K and Q loads; V's flips in the Mm phase
        if (pend_k) ptx::mbar_wait(bar_k, tma_parity, f.a.wait_limit_ns);
        if (pend_q) ptx::mbar_wait(bar_q, tma_parity, f.a.wait_limit_ns);
        if (pend_v) ptx::mbar_wait(bar_v, tma_parity, f.a.wait_limit_ns);
    }
    ptx::tc_fence_before();
    ebar();
}

// ====================================================================================================
// inter-chunk chain: a whole CTA (t = 0..511), all 512 TMEM columns
// ====================================================================================================
// Everything is transposed: TMEM lanes are the 128 columns of the state (dv), so that the state and V_new are A
// operands in TMEM and nothing on the chain goes through shared memory:
//   MMA1  D1[dv][0:64] = (W S)^T, then D1[dv][64:128] = (Gamma.Q S)^T     A = bf16 state, B = W, Q
//   V_new^T = U^T - D1[:, 0:64]  -> bf16 -> TMEM
//   MMA2  D3[dv][dk] = (K'^T V_new)^T,  D1[dv][64:128] += (Aqk V_new)^T            A = V_new, B = K', Aqk
//   S <- gamma^C . S + exp(G_C - G_m) . D3  (fp32, in registers: thread = column, half of dk)  -> bf16 -> TMEM
// A step is two dependent round trips tensor core -> registers -> tensor core (with the operands written to shared
// memory with lanes = dk for all 128 columns: 32 + 16 KB a step, a proxy fence in each trip: 2.3 us a step).
//   warps 0-7  compute: TMEM lane quadrant = warp & 3, half of dk / of the tokens = warp >> 2
//   warp 8 issues the MMAs, warp 9 lane 0 loads the tiles, warps 12-15 write the output rows
// kRing: tiles come from the engines of the cluster; otherwise from the plain array that the intra-chunk kernel
// has written, and `cid` numbers the (sequence, head) pairs.  kRows32 (layer calls): the output rows stay in fp32,
// in the place of the tile's [W ; Q], for the output stage (kda_layer.cu).  kSeg: see SegInfo.
__device__ __forceinline__ float bf16_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf16_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

template <bool kHasQ, bool kRows32, bool kRing, int kSeg = 0>
__device__ void chain_run(const FusedArgs& f, uint8_t* smem, uint32_t tm, int t, int cid, const CUtensorMap* tm_o)
{
    const ChunkArgs& a = f.a;
    uint64_t* ready = reinterpret_cast<uint64_t*>(smem + C_BAR);   // [engine][depth] a ring position holds a tile
    uint64_t* fullA = ready + 6 * kMaxDepth; // [kStagesA] landed
    uint64_t* fullB = fullA + kStagesA;      // [kStagesB]
    uint64_t* emptyA = fullB + kStagesB;     // [kStagesA] MMA1 done with it; kRing: and its landing seen by warp 10
    uint64_t* emptyB = emptyA + kStagesA;    // [kStagesB] last product and the 8 compute warps done with it
    uint64_t* m1 = emptyB + kStagesB;        // MMA1 of a chunk complete
    uint64_t* m2 = m1 + 1;                   // MMA2
    uint64_t* out_bar = m2 + 1;              // [2] output accumulator complete (alternating)
    uint64_t* o_done = out_bar + 2;          // [2] and read (4 warps)
    uint64_t* s_ready = o_done + 2;          // state operand written (8 warps)
    uint64_t* vn_ready = s_ready + 1;        // V_new operand written (8 warps)
    uint64_t* done = vn_ready + 1;           // all MMAs complete, where a wait has run out
    volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(done + 1);
    const int warp = ptx::warp_uniform(t >> 5), lane = t & 31;
    __nv_bfloat16* op = kHasQ ? reinterpret_cast<__nv_bfloat16*>(a.o) : nullptr;

    auto wait_by = [&](auto attempt, uint64_t* bar, uint32_t parity, int where) {
        if (attempt(bar, parity)) return;        // (one access to the busy shared memory where one will do)
        if (*abort_flag) return;
        const uint64_t t0 = ptx::globaltimer_ns();
        uint32_t spins = 0;
        while (!attempt(bar, parity)) {
            if ((++spins & 15u) == 0) {
                if (*abort_flag) return;
                if (call_aborted(f)) { *abort_flag = 1; return; }
                if (ptx::globaltimer_ns() - t0 > a.wait_limit_ns) {
                    *abort_flag = 1;
                    report(f, KDA_ERR_TIMEOUT, where);
                    return;
                }
            }
        }
    };
    auto wait = [&](uint64_t* bar, uint32_t parity, int where) {
        wait_by([](uint64_t* b, uint32_t p) { return ptx::mbar_try(b, p); }, bar, parity, where);
    };
    auto wait_cluster = [&](uint64_t* bar, uint32_t parity, int where) {
        wait_by([](uint64_t* b, uint32_t p) { return ptx::mbar_try_cluster(b, p); }, bar, parity, where);
    };
    // The flag may change between two lanes' looks at it.  Who goes on together leaves together: a warp by a vote, the output
    // warps by their barrier.
    auto aborted = [&]() { return __any_sync(0xffffffffu, *abort_flag != 0) != 0; };
    auto warp_arrive = [&](uint64_t* bar) {
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(bar);
    };
    JobInfo J;
    auto next_job = [&](int r) { return kRing ? job_info(f, cid, r, J) : pass_job<kSeg>(f, cid, r, J); };

    if (warp < 8) {
        if (!kRing) ptx::reg_inc<kChainRegs>();
        // ================= compute warps =================
        const int quad = warp & 3, half = warp >> 2, dv = quad * 32 + lane, dk0 = half * 64;
        const uint32_t tq = tm + ((uint32_t)(quad * 32) << 16);
        float S[64];
#pragma unroll
        for (int i = 0; i < 64; ++i) S[i] = 0.f;
        uint32_t g = 0;
        KT_DECL(8);
        for (int r = 0; next_job(r); ++r) {
            const size_t s_off = ((size_t)J.n * a.H + J.h) * (size_t)(kD * kD);
            const int s_at = dk0 * kD + dv;
            const float* s_in = state_in<kSeg>(f, s_off, cid);
            const bool unit = seg_info<kSeg>(f, cid).unit;
#pragma unroll
            for (int i = 0; i < 64; ++i) S[i] = s_in ? s_in[s_at + i * kD] : unit && dk0 + i == dv ? 1.f : 0.f;
            const float um = unit ? 0.f : 1.f;
            if (J.nch > 0) {
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    uint32_t z[16];
#pragma unroll
                    for (int i = 0; i < 16; ++i) z[i] = pack_bf16(S[b * 32 + 2 * i], S[b * 32 + 2 * i + 1]);
                    ptx::tmem_st_32x32b_x16(tq + T_S + half * 32 + b * 16, z);
                }
                ptx::tmem_st_wait();
                ptx::tc_fence_before();
                warp_arrive(s_ready);
            }
            for (int c = 0; c < J.nch; ++c, ++g) {
                const uint32_t s = g % kStagesB;
                const uint8_t* sb = smem + C_B + s * C_STAGEB;
                const bool more = c + 1 < J.nch;
                // four values of a gate vector of the chunk (0: gamma^C, 1: exp(G_C - G_m))
                auto vec = [&](int which, int i) {
                    return *reinterpret_cast<const float4*>(sb + B_GV + which * 512 + (dk0 + i) * 4);
                };
                KT_MARK(t == 0, 0);
                wait(&fullB[s], (g / kStagesB) & 1u, 6);
                KT_MARK(t == 0, 1);
                {   // V_new^T = U^T - (W S)^T: column dv, tokens 32 half ..
                    uint4 uq[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k)
                        uq[k] = *reinterpret_cast<const uint4*>(sb + B_U + tc::ut_off((uint32_t)dv, (uint32_t)(half * 4 + k)));
                    const uint32_t* u = reinterpret_cast<const uint32_t*>(uq);
                    wait(m1, g & 1u, 7);
                    __syncwarp();
                    KT_MARK(t == 0, 2);
                    ptx::tc_fence_after();
                    uint32_t y[32], z[16];
                    ptx::tmem_ld_32x32b_x32(tq + T_D1 + (g & 1u) * 128u + half * 32, y);
                    ptx::tmem_ld_wait();
#pragma unroll
                    for (int i = 0; i < 16; ++i)
                        z[i] = kSeg == 1 ? pack_bf16(fmaf(um, bf16_lo(u[i]), -__uint_as_float(y[2 * i])), fmaf(um, bf16_hi(u[i]), -__uint_as_float(y[2 * i + 1])))
                                         : pack_bf16(bf16_lo(u[i]) - __uint_as_float(y[2 * i]), bf16_hi(u[i]) - __uint_as_float(y[2 * i + 1]));
                    ptx::tmem_st_32x32b_x16(tq + T_VN + half * 16, z);
                    ptx::tmem_st_wait();
                    ptx::tc_fence_before();
                    warp_arrive(vn_ready);
                }
                KT_MARK(t == 0, 3);
                // S_new = gamma^C . S + exp(G_C - G_m) . D3; the part that does not need D3 comes before the wait
#pragma unroll
                for (int i = 0; i < 64; i += 4) {
                    const float4 e = vec(0, i);
                    S[i] *= e.x; S[i + 1] *= e.y; S[i + 2] *= e.z; S[i + 3] *= e.w;
                }
                KT_MARK(t == 0, 4);
                wait(m2, g & 1u, 9);
                __syncwarp();
                KT_MARK(t == 0, 5);
                ptx::tc_fence_after();
#pragma unroll
                for (int b = 0; b < 2; ++b) {
                    uint32_t y[32];
                    ptx::tmem_ld_32x32b_x32(tq + T_D3 + dk0 + b * 32, y);
#pragma unroll
                    for (int hb = 0; hb < 2; ++hb) {
                        float4 ct[4];      // (the first fetched while the accumulator is)
#pragma unroll
                        for (int i = 0; i < 4; ++i) ct[i] = vec(1, b * 32 + hb * 16 + 4 * i);
                        if (hb == 0) ptx::tmem_ld_wait();
                        uint32_t z[8];
#pragma unroll
                        for (int i = 0; i < 16; i += 4) {
                            float* s4 = &S[b * 32 + hb * 16 + i];
                            const uint32_t* d = y + hb * 16 + i;
                            const float4 e = ct[i / 4];
                            const float2 lo = __ffma2_rn(make_float2(e.x, e.y), make_float2(__uint_as_float(d[0]), __uint_as_float(d[1])),
                                                         make_float2(s4[0], s4[1]));
                            const float2 hi = __ffma2_rn(make_float2(e.z, e.w), make_float2(__uint_as_float(d[2]), __uint_as_float(d[3])),
                                                         make_float2(s4[2], s4[3]));
                            s4[0] = lo.x; s4[1] = lo.y; s4[2] = hi.x; s4[3] = hi.y;
                            z[i / 2] = pack_bf16(lo.x, lo.y);
                            z[i / 2 + 1] = pack_bf16(hi.x, hi.y);
                        }
                        if (more) ptx::tmem_st_32x32b_x8(tq + T_S + half * 32 + b * 16 + hb * 8, z);
                    }
                }
                if (more) ptx::tmem_st_wait();
                ptx::tc_fence_before();
                __syncwarp();
                if (lane == 0) {
                    if (more) ptx::mbar_arrive(s_ready);
                    ptx::mbar_arrive(&emptyB[s]);
                }
                KT_MARK(t == 0, 6);
            }
            if (aborted()) break;
            if (float* s_out = state_out<kSeg>(f, s_off, cid))
#pragma unroll
                for (int i = 0; i < 64; ++i) s_out[s_at + i * kD] = S[i];
        }
        KT_FLUSH(t == 0, f.hdr, 28, 7);
    } else {
        if (!kRing) ptx::reg_dec<256 - kChainRegs>();
        if (warp == 9) {
            // ================= loader =================
            if (lane == 0) {
                uint32_t g = 0;
                KT_DECL(4);
                for (int r = 0; next_job(r) && !*abort_flag; ++r)
                    for (int c = 0; c < J.nch && !*abort_flag; ++c, ++g) {
                        const uint32_t e = g % (uint32_t)f.n_eng, m = g / (uint32_t)f.n_eng;
                        const uint32_t slot = m % (uint32_t)f.depth, sa = g % kStagesA, s = g % kStagesB;
                        const char* tile = kRing ? f.ring + (size_t)(((uint32_t)cid * f.n_eng + e) * f.depth + slot) * tc::TILE_BYTES
                                                 : f.ring + (size_t)(J.tile0 + (int64_t)c * a.H) * tc::TILE_BYTES;
                        KT_MARK(true, 0);
                        if (kRing) {
                            wait_cluster(&ready[e * (uint32_t)f.depth + slot], (m / (uint32_t)f.depth) & 1u, 30);
                            ptx::fence_async_global();
                        }
                        KT_MARK(true, 1);
                        if (g >= kStagesB) wait(&emptyB[s], (g / kStagesB - 1) & 1u, 32);
                        if (*abort_flag) break;
                        KT_MARK(true, 2);
                        uint8_t* sB = smem + C_B + s * C_STAGEB;
                        if (kHasQ) {
                            ptx::mbar_expect_tx(&fullB[s], kBBytes);
                            ptx::bulk_g2s(sB, tile + tc::OFF_KI, kBBytes, &fullB[s]);
                        } else {   // state-only call: only the W rows exist, and no Aqk
                            ptx::mbar_expect_tx(&fullB[s], kBBytes - 8192);
                            ptx::bulk_g2s(sB, tile + tc::OFF_KI, 16384, &fullB[s]);
                            ptx::bulk_g2s(sB + B_GV, tile + tc::OFF_GV, tc::GV_BYTES + 16384, &fullB[s]);
                        }
                        if (g >= kStagesA) wait(&emptyA[sa], (g / kStagesA - 1) & 1u, 34);
                        uint8_t* sA = smem + C_A + sa * kABytes;
                        if (kHasQ) {
                            ptx::mbar_expect_tx(&fullA[sa], kABytes);
                            ptx::bulk_g2s(sA, tile, kABytes, &fullA[sa]);
                        } else {
                            ptx::mbar_expect_tx(&fullA[sa], 16384);
                            ptx::bulk_g2s(sA, tile, 8192, &fullA[sa]);
                            ptx::bulk_g2s(sA + tc::QW_HALF, tile + tc::QW_HALF, 8192, &fullA[sa]);
                        }
                    }
                KT_FLUSH(true, f.hdr, 24, 3);
                if (*abort_flag) {   // the copies already requested must land before the shared memory goes away
                    for (uint32_t x = g > kStagesB ? g - kStagesB : 0; x < g; ++x)
                        ptx::mbar_wait(&fullB[x % kStagesB], (x / kStagesB) & 1u, a.wait_limit_ns / 8);
                    for (uint32_t x = g > kStagesA ? g - kStagesA : 0; x < g; ++x)
                        ptx::mbar_wait(&fullA[x % kStagesA], (x / kStagesA) & 1u, a.wait_limit_ns / 8);
                }
            }
        } else if (kRing && warp == 10) {
            // ================= gives the ring's positions back =================
            // (the loader has no time for the release arrivals; it refills a stage only after this warp has seen it)
            if (lane == 0) {
                const uint32_t base = ptx::smem_u32(smem);
                uint32_t g = 0;
                for (int r = 0; next_job(r) && !*abort_flag; ++r)
                    for (int c = 0; c < J.nch && !*abort_flag; ++c, ++g) {
                        wait(&fullB[g % kStagesB], (g / kStagesB) & 1u, 31);
                        wait(&fullA[g % kStagesA], (g / kStagesA) & 1u, 33);
                        if (*abort_flag) break;
                        ptx::mbar_arrive(&emptyA[g % kStagesA]);
                        ptx::mbar_arrive(&emptyB[g % kStagesB]);
                        const uint32_t e = g % (uint32_t)f.n_eng, slot = (g / (uint32_t)f.n_eng) % (uint32_t)f.depth;
                        ptx::mbar_arrive_cluster(ptx::map_to_cta(base + (e & 1u) * E_BYTES + E_BAR + 48 + slot * 8, 1 + (e >> 1)));
                    }
            }
        } else if (warp == 8) {
            // ================= MMA issue =================
            const uint32_t id1 = ptx::umma_idesc_bf16(128, 64);
            const uint32_t id2 = ptx::umma_idesc_bf16(128, 128) | ptx::kIdescBMajorMN;
            const uint32_t base = (uint32_t)ptx::warp_uniform((int)ptx::smem_u32(smem));
            uint32_t g = 0;
            KT_DECL(8);
            for (int r = 0; next_job(r) && !aborted(); ++r)
                for (int c = 0; c < J.nch && !aborted(); ++c, ++g) {
                    const uint32_t sa = g % kStagesA, s = g % kStagesB;
                    const uint32_t pA = base + C_A + sa * kABytes, pB = base + C_B + s * C_STAGEB;
                    const uint32_t d1 = tm + T_D1 + (g & 1u) * 128u;
                    KT_MARK(lane == 0, 0);
                    wait(&fullA[sa], (g / kStagesA) & 1u, 1);
                    KT_MARK(lane == 0, 1);   // operands
                    if (op && g >= 2) wait(&o_done[g & 1u], ((g >> 1) - 1) & 1u, 2);
                    wait(s_ready, g & 1u, 3);
                    __syncwarp();
                    KT_MARK(lane == 0, 2);   // state
                    ptx::tc_fence_after();
                    // W S first: V_new waits for it alone, Q S runs beside V_new's arithmetic
    #pragma unroll
                    for (int k = 0; k < 8; ++k)
                        ptx::umma_bf16_ta(d1, tm + T_S + k * 8, ptx::umma_desc_sw128(pA + (k >> 2) * tc::QW_HALF + (k & 3) * 32), id1, k > 0);
                    ptx::umma_commit(m1);
                    if (kHasQ) {
    #pragma unroll
                        for (int k = 0; k < 8; ++k)
                            ptx::umma_bf16_ta(d1 + 64, tm + T_S + k * 8,
                                              ptx::umma_desc_sw128(pA + 8192 + (k >> 2) * tc::QW_HALF + (k & 3) * 32), id1, k > 0);
                    }
                    ptx::umma_commit(&emptyA[sa]);
                    KT_MARK(lane == 0, 3);   // MMA1 issue
                    wait(&fullB[s], (g / kStagesB) & 1u, 11);
                    wait(vn_ready, g & 1u, 4);
                    __syncwarp();
                    KT_MARK(lane == 0, 4);   // V_new
                    ptx::tc_fence_after();
    #pragma unroll
                    for (int k = 0; k < 4; ++k)
                        ptx::umma_bf16_ta(tm + T_D3, tm + T_VN + k * 8, ptx::umma_desc_sw128_mn(pB + B_KI + k * 2048, tc::KI_HALF), id2, k > 0);
                    ptx::umma_commit(m2);
                    if (op) {
    #pragma unroll
                        for (int k = 0; k < 4; ++k)
                            ptx::umma_bf16_ta(d1 + 64, tm + T_VN + k * 8, ptx::umma_desc_sw128(pB + B_AQ + k * 32), id1, 1);
                        ptx::umma_commit(&out_bar[g & 1u]);
                    }
                    ptx::umma_commit(&emptyB[s]);
                    KT_MARK(lane == 0, 5);   // MMA2 + output issue
                }
            KT_FLUSH(lane == 0, f.hdr, 16, 6);
            // every MMA has completed before the TMEM goes away
            if (g > 0) wait(&emptyB[(g - 1) % kStagesB], ((g - 1) / kStagesB) & 1u, 5);
            if (aborted()) {
                ptx::umma_commit(done);
                ptx::mbar_wait(done, 0, a.wait_limit_ns);
                __syncwarp();
            }
        } else if (warp >= 12 && op) {
            // ================= output rows =================
            // The accumulator has a lane per column and a TMEM column per token; read as 8 x 8 fragments and stored with
            // stmatrix.trans it becomes rows of the output, which leave by two tiled TMA stores.  (Straight from the lanes, 64 two-byte stores a thread, the stores
            // crowded out the loads of the compute warps: 2.6 instead of 1.6 us a step.)
            const int quad = warp & 3, ot = t - 384;
            const uint32_t tq = tm + ((uint32_t)(quad * 32) << 16);
            // this lane's row of the four 8 x 8 matrices of token block 0, in the swizzled [2][64 tokens][64] image
            const uint32_t mrow = (uint32_t)(lane & 7), mcol = (uint32_t)((quad & 1) * 32 + (lane >> 3) * 8);
            const uint32_t moff = (uint32_t)(quad >> 1) * 8192u + ptx::sw128_off(mrow, mcol);
            uint32_t g = 0;
            bool stop = false;
            for (int r = 0; !stop && next_job(r); ++r)
                for (int c = 0; c < J.nch && !stop; ++c, ++g) {
                    const int64_t tok0 = J.tok_begin + (int64_t)c * kC;
                    const int len = (J.tok_end - tok0) < kC ? (int)(J.tok_end - tok0) : kC;
                    wait(&out_bar[g & 1u], (g >> 1) & 1u, 10);
                    __syncwarp();
                    ptx::tc_fence_after();
                    const uint32_t seen = *abort_flag;      // (looked at beside the read-out: at the barrier it cost a layer call on 24 chains 3 per cent)
                    if (kRows32) {     // lane = column, four tokens a piece
                        uint32_t y[2][32];
                        ptx::tmem_ld_32x32b_x32(tq + T_D1 + (g & 1u) * 128u + 64, y[0]);
                        ptx::tmem_ld_32x32b_x32(tq + T_D1 + (g & 1u) * 128u + 96, y[1]);
                        ptx::tmem_ld_wait();
                        ptx::tc_fence_before();
                        warp_arrive(&o_done[g & 1u]);
                        if (ot == 0) ptx::bulk_wait_read0();      // the previous block has been read out of its buffer
                        stop = ptx::named_bar_or(6, 128, seen != 0);
                        uint4* rows = reinterpret_cast<uint4*>(smem + C_OUT) + ot;
    #pragma unroll
                        for (int q = 0; q < 16; ++q)
                            rows[q * 128] = make_uint4(y[q >> 3][4 * (q & 7)], y[q >> 3][4 * (q & 7) + 1], y[q >> 3][4 * (q & 7) + 2],
                                                       y[q >> 3][4 * (q & 7) + 3]);
                        ptx::fence_async_smem();
                        ptx::named_bar_sync(6, 128);
                        if (ot == 0 && !*abort_flag) {
                            ptx::bulk_s2g(f.ring + (size_t)(J.tile0 + (int64_t)c * a.H) * tc::TILE_BYTES + tc::OFF_O32, smem + C_OUT, 32768);
                            ptx::bulk_commit();
                        }
                        continue;
                    }
                    // y[b >> 1][4 j + 2 (b & 1) + e]: column 8 b + lane / 4 of the quadrant, token 8 j + 2 (lane % 4) + e
                    uint32_t y[2][32];
                    ptx::tmem_ld_16x256b_x8(tq + T_D1 + (g & 1u) * 128u + 64, y[0]);
                    ptx::tmem_ld_16x256b_x8(tq + (16u << 16) + T_D1 + (g & 1u) * 128u + 64, y[1]);
                    ptx::tmem_ld_wait();
                    ptx::tc_fence_before();
                    warp_arrive(&o_done[g & 1u]);
                    // the previous block has been read out of its buffer
                    uint8_t* sb = smem + C_OUT;
                    if (ot == 0) ptx::bulk_wait_read0();
                    stop = ptx::named_bar_or(6, 128, seen != 0);
    #pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        uint32_t z[4];
    #pragma unroll
                        for (int b = 0; b < 4; ++b)
                            z[b] = pack_bf16(__uint_as_float(y[b >> 1][4 * j + 2 * (b & 1)]), __uint_as_float(y[b >> 1][4 * j + 2 * (b & 1) + 1]));
                        ptx::stmatrix_x4_trans(sb + moff + j * 1024, z);
                    }
                    ptx::fence_async_smem();
                    ptx::named_bar_sync(6, 128);
                    if (len == kC) {
                        if (ot == 0 && !*abort_flag) {
                            ptx::tma_store_2d(tm_o, sb, J.h * kD, (int)tok0);
                            ptx::tma_store_2d(tm_o, sb + 8192, J.h * kD + 64, (int)tok0);
                            ptx::bulk_commit();
                        }
                    } else {       // the rows past the end of the sequence belong to the next one
                        if (!*abort_flag)
                            for (int idx = ot; idx < len * 16; idx += 128) {
                                const int row = idx >> 4, ch = idx & 15;
                                *reinterpret_cast<uint4*>(op + ((size_t)(tok0 + row) * a.H + J.h) * kD + ch * 8) =
                                    *reinterpret_cast<const uint4*>(sb + (ch >> 3) * 8192 + ptx::sw128_off((uint32_t)row, (uint32_t)(ch & 7) * 8));
                            }
                    }
                }
            if (ot == 0) ptx::bulk_wait_all0();
        }
    }
    ptx::tc_fence_before();
    __syncthreads();
}

// barriers of a chain CTA; ONE thread
__device__ void chain_init(uint8_t* smem, int ring)
{
    uint64_t* b = reinterpret_cast<uint64_t*>(smem + C_BAR);
    for (int i = 0; i < 6 * kMaxDepth; ++i) ptx::mbar_init(b++, 1);   // ready
    for (int i = 0; i < kStagesA + kStagesB; ++i) ptx::mbar_init(b++, 1);   // fullA, fullB
    for (int i = 0; i < kStagesA; ++i) ptx::mbar_init(b++, 1 + ring);   // emptyA
    for (int i = 0; i < kStagesB; ++i) ptx::mbar_init(b++, 9 + ring);   // emptyB
    ptx::mbar_init(b++, 1);                                           // m1
    ptx::mbar_init(b++, 1);                                           // m2
    for (int i = 0; i < 2; ++i) ptx::mbar_init(b++, 1);               // out_bar
    for (int i = 0; i < 2; ++i) ptx::mbar_init(b++, 4);               // o_done
    ptx::mbar_init(b++, 8);                                           // s_ready
    ptx::mbar_init(b++, 8);                                           // vn_ready
    ptx::mbar_init(b++, 1);                                           // done
    *reinterpret_cast<volatile uint32_t*>(b) = 0;                     // abort flag
    ptx::fence_mbar_init();
}

// One cluster = a chain CTA (rank 0) and CTAs of two engines each; ring positions are handed over by
// mbarriers in each other's shared memory.  The ring is written and read by bulk copies alone: an engine
// announces a tile once its copies have completed, the chain gives a position back once its copy has landed; both
// by release arrivals, taken up by acquire waits and a proxy fence before the next bulk copy.  The arrivals are made where
// nothing waits for the thread, during the substitution and by a warp of their own: 4096 x 32 heads 120.7 us when they were
// added, 1 Mi tokens for the state 20.6 ms, 114 and 20.1 now (made by the loader, and by the service thread ahead of its copies, then: 141 us
// and 28.9 ms; relaxed, which orders nothing, then: 112.5 and 20.2).
template <bool kHasQ>
__global__ void __launch_bounds__(kThreads, 1)
kda_fused_tc(const __grid_constant__ FusedArgs f, const __grid_constant__ CUtensorMap tm_k,
             const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_v,
             const __grid_constant__ CUtensorMap tm_o)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    const int t = threadIdx.x, warp = t >> 5;
    // (from blockIdx and not from %cluster_ctarank: a branch that the compiler does not know to be uniform costs the
    // MMA-issuing warps their uniform registers, 381 instead of 85 ns for the first product of a step)
    const int cid = (int)blockIdx.x / f.cluster_size, rank = (int)blockIdx.x - cid * f.cluster_size;
    const bool chain_cta = rank == 0;
    // (the TMEM slot sits in a spare word of the barrier block of either layout)
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + (chain_cta ? C_BAR + 500 : E_BAR + 32));
    if (chain_cta && t == 0) chain_init(smem, 1);
    if (!chain_cta && (t == 0 || t == kEngThreads)) {
        uint64_t* mb = reinterpret_cast<uint64_t*>(smem + (t ? E_BYTES : 0) + E_BAR);
        ptx::mbar_init(mb, 2);       // MMA group complete (two issuing warps)
        ptx::mbar_init(mb + 1, 1);   // k landed
        ptx::mbar_init(mb + 3, 1);   // q landed
        ptx::mbar_init(mb + 5, 1);   // v landed
        for (int i = 0; i < kMaxDepth; ++i) ptx::mbar_init(mb + 6 + i, 1);   // ring positions free
        *reinterpret_cast<volatile uint32_t*>(mb + 2) = 0;
        ptx::fence_mbar_init();
        if (t == 0) {
            ptx::prefetch_tmap(&tm_k);
            ptx::prefetch_tmap(&tm_q);
            ptx::prefetch_tmap(&tm_v);
        }
    }
    if (warp == 0) {
        ptx::tmem_alloc(tmem_slot, kTmemCols);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::cluster_sync_all();      // every CTA's barriers exist before anybody arrives on them
    ptx::tc_fence_after();
    ptx::grid_dep_wait();         // (launched before the preceding kernel has ended)
    ptx::grid_dep_launch();
    if (blockIdx.x == 0 && t == 0) {
        f.hdr->status = 0;
        f.hdr->where = 0;
        f.hdr->flags = 0;
    }
    const uint32_t tmem_base = (uint32_t)ptx::warp_uniform((int)*tmem_slot);
    if ((ptx::smem_u32(smem) & 1023u) != 0) {   // the operand images need 1024-byte alignment
        if (t == 0) report(f, KDA_ERR_CUDA, 90);
    } else if (chain_cta) {
        chain_run<kHasQ, false, true>(f, smem, tmem_base, t, cid, &tm_o);
    } else {
        const int sub = ptx::warp_uniform(t / kEngThreads), e = (rank - 1) * 2 + sub;
        if (e < f.n_eng) {
            uint8_t* es = smem + sub * E_BYTES;
            if (t - sub * kEngThreads == kServiceThread)
                *reinterpret_cast<EngineCursor*>(es + E_CUR) = {
                    cid, e, 0, e, 0, ptx::map_to_cta(ptx::smem_u32(smem) + C_BAR + (uint32_t)(e * f.depth) * 8u, 0), 0, 0};
            engine_run<kHasQ, true>(f, es, tmem_base + sub * 256, 1 + sub, t - sub * kEngThreads, 0, 0, &tm_k, &tm_q, &tm_v);
        }
    }
    ptx::tc_fence_before();
    __syncthreads();
    if (warp == 0) ptx::tmem_dealloc(tmem_base, kTmemCols);
    ptx::cluster_sync_all();      // no CTA leaves while another may still arrive on its barriers
}

// ---- the chains alone (second kernel of the two-kernel schedule): a CTA per (sequence, head) -------------------
template <bool kHasQ, bool kRows32, int kSeg>
__global__ void __launch_bounds__(kThreads, 1)
kda_chain_tc(const __grid_constant__ FusedArgs f, const __grid_constant__ CUtensorMap tm_o)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    const int t = threadIdx.x, warp = t >> 5;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + C_BAR + 500);
    if (t == 0) chain_init(smem, 0);
    if (warp == 0) {
        ptx::tmem_alloc(tmem_slot, kTmemCols);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem_base = (uint32_t)ptx::warp_uniform((int)*tmem_slot);
    if ((ptx::smem_u32(smem) & 1023u) != 0) {
        if (t == 0) report(f, KDA_ERR_CUDA, 90);
    } else {
        // The tiles, the chunk table and S0 come from kernels before this one.  Only then the next may start: what
        // that reads before its own wait (the gates of kda_layer_rows_kernel) is older than this kernel's inputs.
        ptx::grid_dep_wait();
        ptx::grid_dep_launch();
        chain_run<kHasQ, kRows32, false, kSeg>(f, smem, tmem_base, t, (int)blockIdx.x, &tm_o);
    }
    ptx::tc_fence_before();
    __syncthreads();
    if (warp == 0) ptx::tmem_dealloc(tmem_base, kTmemCols);
}

// ---- the intra-chunk stage alone (first kernel of the two-kernel schedule) --------------------------------
// Persistent CTAs of one engine each, two per SM; the tiles of the pass go to a plain array.
template <bool kHasQ, bool kLayer>
__global__ void __launch_bounds__(kEngThreads, 2)
kda_intra_tc(const __grid_constant__ FusedArgs f, const __grid_constant__ CUtensorMap tm_k,
             const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_v,
             int clear_status)
{
    extern __shared__ __align__(1024) uint8_t smem[];
    const int t = threadIdx.x, warp = t >> 5;
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem + E_BAR + 32);
    if (t == 0) {
        uint64_t* mb = reinterpret_cast<uint64_t*>(smem + E_BAR);
        ptx::mbar_init(mb, 2);       // MMA group complete (two issuing threads)
        ptx::mbar_init(mb + 1, 1);   // k landed
        ptx::mbar_init(mb + 3, 1);   // q landed
        ptx::mbar_init(mb + 5, 1);   // v landed
        *reinterpret_cast<volatile uint32_t*>(mb + 2) = 0;
        ptx::fence_mbar_init();
        ptx::prefetch_tmap(&tm_k);
        ptx::prefetch_tmap(&tm_q);
        ptx::prefetch_tmap(&tm_v);
    }
    if (warp == 0) {
        ptx::tmem_alloc(tmem_slot, 256);
        ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tmem_base = (uint32_t)ptx::warp_uniform((int)*tmem_slot);
    if ((ptx::smem_u32(smem) & 1023u) != 0) {
        if (t == 0) report(f, KDA_ERR_CUDA, 90);   // the operand images need 1024-byte alignment
    } else {
        ptx::grid_dep_wait();     // (launched before the preceding kernel has ended)
        ptx::grid_dep_launch();   // the chains may set themselves up while this one drains
        if (clear_status && blockIdx.x == 0 && t == 0) {
            f.hdr->status = 0;      // (an equal-length call has no prologue kernel to do this)
            f.hdr->where = 0;
            f.hdr->flags = 0;
        }
        engine_run<kHasQ, false, kLayer>(f, smem, tmem_base, 1, t, blockIdx.x, gridDim.x, &tm_k, &tm_q, &tm_v);
    }
    ptx::tc_fence_before();
    __syncthreads();
    if (warp == 0) ptx::tmem_dealloc(tmem_base, 256);
}

// cuTensorMapEncodeTiled through the runtime's driver entry-point query (no link dependency on
// libcuda, so the library still loads on a machine without a driver)
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);
EncodeTiledFn get_encode_fn()
{
    static EncodeTiledFn fn = nullptr;   // (the entry point is the same for every device: benign race)
    if (!fn) {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult qres;
        if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &qres) == cudaSuccess &&
            qres == cudaDriverEntryPointSuccess)
            fn = reinterpret_cast<EncodeTiledFn>(p);
    }
    return fn;
}
// [total_tokens, H*128] bf16 matrix, boxes of 64 tokens x 64 channels, 128-byte swizzle
kda_status_t make_tmap(CUtensorMap* tm, const void* base, int64_t total_tokens, int H)
{
    EncodeTiledFn fn = get_encode_fn();
    if (!fn) return fail(KDA_ERR_CUDA, "cuTensorMapEncodeTiled is not available from the driver");
    const cuuint64_t dims[2] = {(cuuint64_t)H * kD, (cuuint64_t)total_tokens};
    const cuuint64_t strides[1] = {(cuuint64_t)H * kD * 2};
    const cuuint32_t box[2] = {64, 64};
    const cuuint32_t estr[2] = {1, 1};
    CUresult r = fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box,
                    estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                    CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) return fail(KDA_ERR_CUDA, "cuTensorMapEncodeTiled failed with code %d", (int)r);
    return KDA_OK;
}

}  // namespace

kda_status_t launch_intra_tc(const ChunkArgs& a, void* tiles, WsHeader* hdr, bool clear_status,
                             cudaStream_t st)
{
    int n_sm = 0;
    {
        DeviceLock lk;
        if (!lk.st) return lk.rc;
        if (!lk.st->attr_done[1]) {
            KDA_CUDA_TRY(cudaFuncSetAttribute(kda_intra_tc<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)E_BYTES));
            KDA_CUDA_TRY(cudaFuncSetAttribute(kda_intra_tc<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)E_BYTES));
            KDA_CUDA_TRY(cudaFuncSetAttribute(kda_intra_tc<true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)E_BYTES));
            KDA_CUDA_TRY(cudaFuncSetAttribute(kda_intra_tc<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)E_BYTES));
            lk.st->attr_done[1] = true;
        }
        if (lk.st->n_sm == 0) {
            int dev = 0;
            KDA_CUDA_TRY(cudaGetDevice(&dev));
            KDA_CUDA_TRY(cudaDeviceGetAttribute(&lk.st->n_sm, cudaDevAttrMultiProcessorCount, dev));
        }
        n_sm = lk.st->n_sm;
    }
    const int64_t n_tiles = (a.g1 - a.g0) * a.H;
    if (n_tiles <= 0) return KDA_OK;
    if (n_tiles > 0x7fffffff || a.total_tokens > 0x7fffffff)
        return fail(KDA_ERR_UNSUPPORTED, "kda_chunk_fwd: more than 2^31 tokens or tiles in one pass");
    FusedArgs f = {};
    f.a = a;
    f.ring = static_cast<char*>(tiles);
    f.hdr = hdr;
    f.n_prod = (uint32_t)n_tiles;
    const bool has_q = a.q != nullptr && a.o != nullptr;
    CUtensorMap tm_k, tm_q, tm_v;
    kda_status_t rc = make_tmap(&tm_k, a.k, a.total_tokens, a.H);
    if (rc == KDA_OK) rc = make_tmap(&tm_v, a.v, a.total_tokens, a.H);
    if (rc == KDA_OK) rc = make_tmap(&tm_q, has_q ? a.q : a.k, a.total_tokens, a.H);
    if (rc != KDA_OK) return rc;
    const int64_t resident = 2 * (int64_t)n_sm;   // two CTAs per SM
    const unsigned grid = (unsigned)(n_tiles < resident ? n_tiles : resident);
    ProfScope ps(PROF_INTRA, st);
    const bool layer = a.gate_rate != nullptr;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(kEngThreads);
    cfg.dynamicSmemBytes = E_BYTES;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    auto fn = layer ? (has_q ? kda_intra_tc<true, true> : kda_intra_tc<false, true>)
                    : (has_q ? kda_intra_tc<true, false> : kda_intra_tc<false, false>);
    KDA_CUDA_TRY(cudaLaunchKernelEx(&cfg, fn, f, tm_k, tm_q, tm_v, clear_status ? 1 : 0));
    count_launch();
    KDA_CUDA_TRY(cudaGetLastError());
    return KDA_OK;
}

namespace {
using FusedFn = void (*)(FusedArgs, CUtensorMap, CUtensorMap, CUtensorMap, CUtensorMap);
using ChainFn = void (*)(FusedArgs, CUtensorMap);
FusedFn fused_fn(bool has_q) { return has_q ? kda_fused_tc<true> : kda_fused_tc<false>; }
ChainFn chain_fn(bool has_q, bool rows32, int seg)
{
    if (seg == 1) return kda_chain_tc<false, false, 1>;
    if (!has_q) return kda_chain_tc<false, false, 0>;
    if (seg == 2) return rows32 ? kda_chain_tc<true, true, 2> : kda_chain_tc<true, false, 2>;
    return rows32 ? kda_chain_tc<true, true, 0> : kda_chain_tc<true, false, 0>;
}
void fused_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute (&at)[2], int cluster, int n_clusters, cudaStream_t st)
{
    cfg = cudaLaunchConfig_t{};
    cfg.gridDim = dim3((unsigned)(cluster * n_clusters));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmemBytes;
    cfg.stream = st;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)cluster; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
}
}  // namespace

// Resident clusters of 3 and of 4 CTAs on the current device (asked once per device).
kda_status_t fused_max_clusters(int (&n)[2])
{
    DeviceLock lk;
    if (!lk.st) return lk.rc;
    if (!lk.st->attr_done[0]) {
        for (int i = 0; i < 2; ++i)
            KDA_CUDA_TRY(cudaFuncSetAttribute((const void*)fused_fn(i), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)kSmemBytes));
        for (int i = 0; i < 2; ++i) {
            cudaLaunchConfig_t cfg;
            cudaLaunchAttribute at[2];
            fused_config(cfg, at, 3 + i, 1, nullptr);
            cfg.numAttrs = 1;
            int c = 0;
            KDA_CUDA_TRY(cudaOccupancyMaxActiveClusters(&c, (const void*)fused_fn(true), &cfg));
            lk.st->fused_clusters[i] = c;
        }
        lk.st->attr_done[0] = true;
    }
    n[0] = lk.st->fused_clusters[0];
    n[1] = lk.st->fused_clusters[1];
    return KDA_OK;
}

kda_status_t launch_fused_tc(const FusedArgs& f, bool has_q, cudaStream_t st)
{
    if (f.a.total_tokens > 0x7fffffff)
        return fail(KDA_ERR_UNSUPPORTED, "kda_chunk_fwd: more than 2^31 tokens in one call");
    const int64_t T = f.a.total_tokens > 0 ? f.a.total_tokens : 1;   // (a call of empty sequences loads nothing)
    const void* any = f.a.k ? f.a.k : f.hdr;
    CUtensorMap tm_k, tm_q, tm_v, tm_o;
    kda_status_t rc = make_tmap(&tm_k, any, T, f.a.H);
    if (rc == KDA_OK) rc = make_tmap(&tm_v, f.a.v ? f.a.v : any, T, f.a.H);
    if (rc == KDA_OK) rc = make_tmap(&tm_q, has_q ? f.a.q : any, T, f.a.H);
    if (rc == KDA_OK) rc = make_tmap(&tm_o, has_q ? f.a.o : any, T, f.a.H);
    if (rc != KDA_OK) return rc;
    cudaLaunchConfig_t cfg;
    cudaLaunchAttribute at[2];
    fused_config(cfg, at, f.cluster_size, f.n_clusters, st);
    ProfScope ps(PROF_FUSED, st);
    KDA_CUDA_TRY(cudaLaunchKernelEx(&cfg, fused_fn(has_q), f, tm_k, tm_q, tm_v, tm_o));
    count_launch();
    return KDA_OK;
}

// second kernel of the two-kernel schedule, for n_count sequences (f.n_begin .., or by f.order)
kda_status_t launch_chain_tc(const FusedArgs& f, int n_count, cudaStream_t st)
{
    const ChunkArgs& a = f.a;
    const bool maps = f.seg_mode == 1, has_q = a.q != nullptr && a.o != nullptr && !maps;
    {
        DeviceLock lk;
        if (!lk.st) return lk.rc;
        if (!lk.st->attr_done[2]) {
            for (int i = 0; i < 12; ++i)
                KDA_CUDA_TRY(cudaFuncSetAttribute((const void*)chain_fn(i & 1, i & 2, i / 4), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                  (int)kSmemBytes));
            lk.st->attr_done[2] = true;
        }
    }
    CUtensorMap tm_o;
    const kda_status_t rc = make_tmap(&tm_o, has_q ? a.o : f.hdr, a.total_tokens > 0 ? a.total_tokens : 1, a.H);
    if (rc != KDA_OK) return rc;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)n_count * (unsigned)a.H * (unsigned)(maps ? f.seg_runs : f.seg_mode ? f.seg_P : 1));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = kSmemBytes;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    // set up beside this library's own intra-chunk kernel
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = a.g1 > a.g0 && f.seg_mode != 2 ? 1 : 0;
    ProfScope ps(PROF_INTER, st);
    KDA_CUDA_TRY(cudaLaunchKernelEx(&cfg, chain_fn(has_q, a.rows32, f.seg_mode), f, tm_o));
    count_launch();
    return KDA_OK;
}

namespace {
// Self-test of the bounded-wait path: one CTA waits on an mbarrier that nothing ever arrives on,
// with a short limit, and must come back with KDA_ERR_TIMEOUT in the status word.
__global__ void kda_wait_selftest_kernel(WsHeader* hdr, uint64_t limit_ns)
{
    __shared__ uint64_t bar;
    if (threadIdx.x == 0) {
        ptx::mbar_init(&bar, 1);
        ptx::fence_mbar_init();
    }
    __syncthreads();
    if (!ptx::mbar_wait(&bar, 0, limit_ns)) {
        if (atomicCAS(&hdr->status, 0, (int)KDA_ERR_TIMEOUT) == 0) hdr->where = 99;
    }
}
}  // namespace

kda_status_t launch_wait_selftest(WsHeader* hdr, uint64_t limit_ns, cudaStream_t st)
{
    kda_wait_selftest_kernel<<<1, 32, 0, st>>>(hdr, limit_ns);
    count_launch();
    KDA_CUDA_TRY(cudaGetLastError());
    return KDA_OK;
}

size_t tc_tile_bytes() { return tc::TILE_BYTES; }

}  // namespace kda
