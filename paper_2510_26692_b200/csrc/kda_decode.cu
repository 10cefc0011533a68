// Recurrent decode step of KDA (paper Section 3, Eq. 1, one token per sequence and head):
//     Sd = Diag(alpha) S;  r = v - Sd^T k;  S = Sd + beta k r^T;  o = scale S^T q
// evaluated in ONE pass over the 128x128 fp32 state using the identity
//     o = scale (Sd^T q + beta (q.k) r),
// so that both column reductions (Sd^T k and Sd^T q) are taken while the state streams through
// registers, and the state is written back exactly once.  HBM-bound: 64 KiB read + 64 KiB written
// per (sequence, head).
//
// One CTA of 256 threads owns one state, or half of its columns (decode_cols).  Of a whole state thread (warp w,
// lane l) holds rows w, w+8, ... and the four columns 4l..4l+3 of each: every warp-level access is one fully coalesced 512-byte row, and
// all 16 loads of a thread are issued before the first use (64 KiB in flight per CTA).
#include "kda_common.cuh"
#include "kda_ptx.cuh"

namespace kda {
namespace {

__device__ __forceinline__ float4 ld_stream(const float* p) {
    float4 r;
    asm volatile("ld.global.L1::no_allocate.v4.f32 {%0,%1,%2,%3}, [%4];"
                 : "=f"(r.x), "=f"(r.y), "=f"(r.z), "=f"(r.w)
                 : "l"(p));
    return r;
}
__device__ __forceinline__ void st_stream(float* p, float4 x) {
    asm volatile("st.global.L1::no_allocate.v4.f32 [%0], {%1,%2,%3,%4};" ::"l"(p), "f"(x.x),
                 "f"(x.y), "f"(x.z), "f"(x.w)
                 : "memory");
}
// packed fp32 arithmetic (two independent round-to-nearest operations per instruction on sm_100):
// in the multi-token kernel's loop
__device__ __forceinline__ void mul4(float4& x, float a) {
    const float2 aa = make_float2(a, a);
    const float2 lo = __fmul2_rn(make_float2(x.x, x.y), aa), hi = __fmul2_rn(make_float2(x.z, x.w), aa);
    x = make_float4(lo.x, lo.y, hi.x, hi.y);
}
__device__ __forceinline__ void fma4(float4& acc, float a, const float4& x) {   // acc += a * x
    const float2 aa = make_float2(a, a);
    const float2 lo = __ffma2_rn(aa, make_float2(x.x, x.y), make_float2(acc.x, acc.y));
    const float2 hi = __ffma2_rn(aa, make_float2(x.z, x.w), make_float2(acc.z, acc.w));
    acc = make_float4(lo.x, lo.y, hi.x, hi.y);
}
template <typename T> __device__ __forceinline__ float to_f(T x);
template <> __device__ __forceinline__ float to_f<float>(float x) { return x; }
template <> __device__ __forceinline__ float to_f<__nv_bfloat16>(__nv_bfloat16 x) {
    return __bfloat162float(x);
}
template <typename T> __device__ __forceinline__ T from_f(float x);
template <> __device__ __forceinline__ float from_f<float>(float x) { return x; }
template <> __device__ __forceinline__ __nv_bfloat16 from_f<__nv_bfloat16>(float x) { return __float2bfloat16_rn(x); }

// Layer mode (kda_layer_decode_step, paper Section 4 "Neural Parameterization"): q and k arrive
// un-normalised, `log_alpha` points to the bf16 pre-activations of the decay function, `beta` to the
// pre-activations of beta, and the output row goes through the head-wise RMSNorm and the sigmoid
// output gate before it is stored.  All of it is arithmetic on 128-vectors beside a 64 KiB state
// stream: free at the HBM bound.
struct DecodeLayer {
    const float* A_log;        // [H]
    const float* dt_bias;      // [H, dk]
    const void* g_o;           // bf16 [n_seqs, H, dv]
    const float* rms_weight;   // [dv]
    float l2_eps, rms_eps;
};

// Columns of the state never mix, so a state may also be cut into column slices of NC columns with a CTA
// each (decode_cols() says when): the lanes of a warp then cover 128 / NC rows at once.  The layer mode's
// RMSNorm needs the whole output row, so it keeps whole states.
template <typename T, bool kLayer, int NC>
__global__ void __launch_bounds__(256, kD / NC * 2)
kda_decode_kernel(const T* q, const T* k, const T* v, const float* log_alpha, const float* beta, float* S,
                  const int32_t* slot, T* o, int H, float scale, DecodeLayer lay)
{
    static_assert(!kLayer || NC == kD, "the output stage needs the whole row");
    constexpr int kSlices = kD / NC;
    constexpr int LPR = NC / 4;              // lanes per row
    constexpr int RPW = 32 / LPR;            // rows of one warp-level access
    constexpr int NX = kD / (8 * RPW);       // rows per thread
    __shared__ float s_a[kD], s_k[kD], s_q[kD];
    __shared__ float4 s_red[2][8][LPR];
    const int item = blockIdx.x / kSlices, slice = blockIdx.x - item * kSlices;
    const int n = item / H, h = item - n * H;
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int col = slice * NC + (lane % LPR) * 4, row0 = warp * RPW + lane / LPR;
    ptx::grid_dep_wait();                    // (launched before the preceding kernel has ended)
    ptx::grid_dep_launch();
    const size_t sl = slot ? (size_t)slot[n] : (size_t)n;
    float* Sp = S + (sl * H + h) * (size_t)(kD * kD) + col;

    // q, k and the decay first: their arithmetic is done by the time the state has arrived.  v and beta, needed at the end, behind
    // the state (12 x 32 states in fp32 7.84 -> 7.75 us, 40 x 32 23.8 -> 23.4; in layer mode, where the gates come too, slower: 37 x 32
    // 24.9 -> 26.0).
    const size_t vec = (size_t)item * kD;
    float b_in = 0.f;
    float4 vv = make_float4(0.f, 0.f, 0.f, 0.f);
    auto request_v = [&]() {
        b_in = beta[item];
        vv = IO<T>::load4(v + vec + col);
    };
    if (kLayer) request_v();
    float4 w4 = make_float4(0.f, 0.f, 0.f, 0.f), g4 = w4;   // for the output stage
    float kv_in = 0.f, qv_in = 0.f, g_in = 0.f, bias_in = 0.f, rate_in = 0.f;
    if (t < kD) {
        kv_in = to_f<T>(k[vec + t]);
        qv_in = to_f<T>(q[vec + t]);
        if (kLayer) {
            g_in = to_f<T>(reinterpret_cast<const T*>(log_alpha)[vec + t]);
            bias_in = lay.dt_bias[(size_t)h * kD + t];
            rate_in = lay.A_log[h];
        } else {
            g_in = log_alpha[vec + t];
        }
    }
    if (kLayer && warp == 0) {
        w4 = *reinterpret_cast<const float4*>(lay.rms_weight + col);
        g4 = IO<T>::load4(reinterpret_cast<const T*>(lay.g_o) + vec + col);
    }
    asm volatile("" ::: "memory");
    float4 x[NX];
#pragma unroll
    for (int m = 0; m < NX; ++m) x[m] = ld_stream(Sp + (size_t)(row0 + 8 * RPW * m) * kD);
    if (!kLayer) request_v();

    if (t < kD) {
        if (kLayer) {
            const float z = g_in + bias_in;
            const float sp = fmaxf(z, 0.f) + log1pf(expf(-fabsf(z)));
            s_a[t] = expf(-expf(rate_in) * sp);
        } else {
            s_a[t] = expf(g_in);
        }
        s_k[t] = kv_in;
        s_q[t] = qv_in;
    }
    __syncthreads();

    // q.k, redundantly per warp (4 rows per lane, butterfly reduce); layer mode: the norms as well
    float qk = 0.f, ssk = 0.f, ssq = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const float kv = s_k[lane * 4 + i], qv = s_q[lane * 4 + i];
        qk += qv * kv;
        if (kLayer) {
            ssk += kv * kv;
            ssq += qv * qv;
        }
    }
#pragma unroll
    for (int ofs = 16; ofs > 0; ofs >>= 1) {
        qk += __shfl_xor_sync(0xffffffffu, qk, ofs);
        if (kLayer) {
            ssk += __shfl_xor_sync(0xffffffffu, ssk, ofs);
            ssq += __shfl_xor_sync(0xffffffffu, ssq, ofs);
        }
    }
    const float rk = kLayer ? rsqrtf(ssk + lay.l2_eps) : 1.f;   // 1 / |k|, 1 / |q| (L2Norm)
    const float rq = kLayer ? rsqrtf(ssq + lay.l2_eps) : 1.f;
    if (kLayer) qk *= rk * rq;

    float4 p = make_float4(0.f, 0.f, 0.f, 0.f), s = p;
#pragma unroll
    for (int m = 0; m < NX; ++m) {
        const int row = row0 + 8 * RPW * m;
        const float a = s_a[row], kk = kLayer ? s_k[row] * rk : s_k[row], qq = kLayer ? s_q[row] * rq : s_q[row];
        x[m].x *= a; x[m].y *= a; x[m].z *= a; x[m].w *= a;
        p.x += kk * x[m].x; p.y += kk * x[m].y; p.z += kk * x[m].z; p.w += kk * x[m].w;
        s.x += qq * x[m].x; s.y += qq * x[m].y; s.z += qq * x[m].z; s.w += qq * x[m].w;
    }
#pragma unroll
    for (int ofs = LPR; ofs < 32; ofs <<= 1) {
        p.x += __shfl_xor_sync(0xffffffffu, p.x, ofs); p.y += __shfl_xor_sync(0xffffffffu, p.y, ofs);
        p.z += __shfl_xor_sync(0xffffffffu, p.z, ofs); p.w += __shfl_xor_sync(0xffffffffu, p.w, ofs);
        s.x += __shfl_xor_sync(0xffffffffu, s.x, ofs); s.y += __shfl_xor_sync(0xffffffffu, s.y, ofs);
        s.z += __shfl_xor_sync(0xffffffffu, s.z, ofs); s.w += __shfl_xor_sync(0xffffffffu, s.w, ofs);
    }
    if (lane < LPR) {
        s_red[0][warp][lane] = p;
        s_red[1][warp][lane] = s;
    }
    __syncthreads();
    p = s_red[0][0][lane % LPR];
#pragma unroll
    for (int w = 1; w < 8; ++w) {   // fixed order: bitwise reproducible
        const float4 a = s_red[0][w][lane % LPR];
        p.x += a.x; p.y += a.y; p.z += a.z; p.w += a.w;
    }
    const float bt = kLayer ? 1.f / (1.f + expf(-b_in)) : b_in;
    const float4 r = make_float4(vv.x - p.x, vv.y - p.y, vv.z - p.z, vv.w - p.w);
#pragma unroll
    for (int m = 0; m < NX; ++m) {
        const int row = row0 + 8 * RPW * m;
        const float c = kLayer ? bt * s_k[row] * rk : bt * s_k[row];
        x[m].x += c * r.x; x[m].y += c * r.y; x[m].z += c * r.z; x[m].w += c * r.w;
        st_stream(Sp + (size_t)row * kD, x[m]);
    }
    // output row: warp 0 (its lanes below LPR)
    float4 ov = make_float4(0.f, 0.f, 0.f, 0.f);
    float ss = 0.f;
    if (warp == 0) {
        s = s_red[1][0][lane % LPR];
#pragma unroll
        for (int w = 1; w < 8; ++w) {
            const float4 b = s_red[1][w][lane % LPR];
            s.x += b.x; s.y += b.y; s.z += b.z; s.w += b.w;
        }
        const float c = bt * qk;
        ov = make_float4(scale * (s.x + c * r.x), scale * (s.y + c * r.y),
                         scale * (s.z + c * r.z), scale * (s.w + c * r.w));
        if (kLayer) {
            ss = ov.x * ov.x + ov.y * ov.y + ov.z * ov.z + ov.w * ov.w;
#pragma unroll
            for (int ofs = LPR / 2; ofs > 0; ofs >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, ofs);
        }
        if (kLayer) {   // head-wise RMSNorm over the 128 values of the row (4 per lane), weight, sigmoid gate
            const float rstd = rsqrtf(ss * (1.f / kD) + lay.rms_eps);
            ov.x *= rstd * w4.x / (1.f + expf(-g4.x));
            ov.y *= rstd * w4.y / (1.f + expf(-g4.y));
            ov.z *= rstd * w4.z / (1.f + expf(-g4.z));
            ov.w *= rstd * w4.w / (1.f + expf(-g4.w));
        }
        IO<T>::store4(o + vec + col, ov);
    }
}

// State columns per CTA of a call over `items` (sequence, head) pairs: half states, four CTAs per SM, have the
// finer first and last wave; whole states win where one wave of two per SM holds the call (n_sm * 2 items)
// and, by the fewer barriers per byte, in long streams.  Measured (us a step, whole / half): 32 states 3.4 /
// 3.1, 96: 4.3 / 3.8, 160: 6.0 / 5.4, 288: 5.8 / 6.0, 512: 14.0 / 13.2, 1184: 27.8 / 26.4, 2048: 44.6 / 42.9,
// 8192: 165.1 / 165.9 (the line at 40 n_sm lies between these two without a point of its own).
inline int decode_cols(int64_t items, int n_sm)
{
    if (items <= n_sm + n_sm / 2) return 64;
    return items <= 2 * n_sm || items > 40 * n_sm ? kD : 64;
}

// Multi-token decode: the same recurrence for T consecutive tokens of each sequence (speculative
// decoding, continuation of a chunked prefill by a few tokens) with the state held in registers
// across the tokens: it crosses HBM once in each direction per call instead of once per token.
// Layout: q, k, log_alpha [n_seqs, T, H, 128], v, o [n_seqs, T, H, 128], beta [n_seqs, T, H].
// Thread layout of the multi-token kernel: warp w owns the 16 state columns 16w..16w+15 for ALL 128
// dk rows; lane (rg, cg) = (lane >> 2, lane & 3) holds rows rg, rg + 8, ..., rg + 120 and the four
// columns 16w + 4cg .. +3.  The two column reductions of a token (S^T k and S^T q, over the dk rows)
// then stay inside the warp: 16 rows in the thread's registers, the 8 row groups by three
// butterfly shuffles.  No shared-memory reduction and no CTA-wide barrier per token (the
// single-token kernel keeps its fully coalesced row layout: it has no token loop to protect).
//
// The tokens of a state depend on each other, so a CTA that only started to fetch its state when
// it began would leave HBM idle while it computes.  CTAs are therefore persistent (two per SM) and
// fetch the NEXT state into shared memory with asynchronous 16-byte copies while they work on the
// current one; every thread copies exactly the elements it will own into its own slots, so the
// hand-over needs no barrier: a thread waits for its own copies only.
__device__ __forceinline__ void cp_async16(void* dst_smem, const void* src_gmem) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst_smem)),
                 "l"(src_gmem)
                 : "memory");
}
// Dynamic shared memory of the multi-token kernel.  Its token loop takes 0.76 us a token and state on an SM (128 x 32
// states, 8 tokens); 128 packed FMAs a thread and what follows fill no pipe for as long, so it is the chain of loads, sums
// and shuffles that each token ends in.  Vectors in four arrays that a thread reads 16 bytes at a time and sums exchanged
// by halves take 16 loads and 11 shuffles a token and warp, where packed (alpha, k, q, beta k) and a butterfly took 32 and 24:
// 64 x 32 states, 4 tokens 64.2 -> 60.9 us; 128 x 32, 8 tokens 185 -> 169.
template <typename T> struct MultiSmem {
    static constexpr int GT = 8;                        // tokens staged together
    static constexpr int kState = 16 * 256 * 16;        // the prefetched state: element m of thread t at [m][t]
    // alpha, k, q and beta k of a token: dk row 8 m + r at float r * kRow + m, so that the 16 rows of a thread are four
    // 16-byte loads and the eight row groups of a warp lie in different banks
    static constexpr int kRow = 20, kVec = 8 * kRow;
    static constexpr int kAkq = 4 * GT * kVec * 4;
    static constexpr int kV = GT * kD * 4;
    static constexpr int kRawA = GT * kD * 4;           // raw log alpha of the next item's first tokens
    static constexpr int kRawX = GT * kD * (int)sizeof(T);   // raw k / q / v of the same tokens
    static constexpr int oAkq = kState, oV = oAkq + kAkq, oRawA = oV + kV, oRawK = oRawA + kRawA,
                         oRawQ = oRawK + kRawX, oRawV = oRawQ + kRawX, oRawB = oRawV + kRawX,
                         kTotal = oRawB + 64;
};
__device__ __forceinline__ void cp_async4b(void* dst_smem, const void* src_gmem) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst_smem)),
                 "l"(src_gmem)
                 : "memory");
}

template <typename T>
__global__ void __launch_bounds__(256, 2)
kda_decode_multi_kernel(const T* q, const T* k, const T* v, const float* log_alpha, const float* beta, float* S,
                        const int32_t* slot, T* o, int H, int n_tok, float scale,
                        int n_items)
{
    using L = MultiSmem<T>;
    constexpr int GT = L::GT;
    extern __shared__ __align__(16) unsigned char sm[];
    float4* s_next = reinterpret_cast<float4*>(sm);
    float (*s_a)[L::kVec] = reinterpret_cast<float(*)[L::kVec]>(sm + L::oAkq);
    float (*s_k)[L::kVec] = s_a + GT, (*s_q)[L::kVec] = s_k + GT, (*s_bk)[L::kVec] = s_q + GT;
    float (*s_v)[kD] = reinterpret_cast<float(*)[kD]>(sm + L::oV);
    float (*r_a)[kD] = reinterpret_cast<float(*)[kD]>(sm + L::oRawA);
    T (*r_k)[kD] = reinterpret_cast<T(*)[kD]>(sm + L::oRawK);
    T (*r_q)[kD] = reinterpret_cast<T(*)[kD]>(sm + L::oRawQ);
    T (*r_v)[kD] = reinterpret_cast<T(*)[kD]>(sm + L::oRawV);
    float* r_b = reinterpret_cast<float*>(sm + L::oRawB);
    __shared__ float s_b[GT], s_qk[GT];
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int rg = lane >> 2, cg = lane & 3, col = warp * 16 + cg * 4;
    auto at = [](int row) { return (row & 7) * L::kRow + (row >> 3); };
    const int gfirst = n_tok < GT ? n_tok : GT;   // tokens of an item's first group

    auto state_of = [&](int item) {
        const int n = item / H, h = item - n * H;
        const size_t sl = slot ? (size_t)slot[n] : (size_t)n;
        return S + (sl * H + h) * (size_t)(kD * kD) + col;
    };
    // Everything the next item needs first -- its state and the vectors of its first tokens -- is
    // requested with asynchronous copies while the current item is worked on.
    auto fetch = [&](int item) {
        const float* Sp = state_of(item);   // a copy instruction of a warp covers 8 consecutive rows x 64 contiguous bytes
#pragma unroll
        for (int m = 0; m < 16; ++m) cp_async16(&s_next[m * 256 + t], Sp + (size_t)(rg + 8 * m) * kD);
        const int n = item / H, h = item - n * H;
        constexpr int CA = kD * 4 / 16, CX = kD * (int)sizeof(T) / 16;   // 16-byte pieces per token
        for (int idx = t; idx < gfirst * (CA + 3 * CX); idx += 256) {
            const int tok = idx / (CA + 3 * CX), j = idx - tok * (CA + 3 * CX);
            const size_t vec = ((size_t)(n * n_tok + tok) * H + h) * kD;
            if (j < CA) cp_async16(&r_a[tok][j * 4], log_alpha + vec + j * 4);
            else if (j < CA + CX) cp_async16(&r_k[tok][(j - CA) * (16 / (int)sizeof(T))], k + vec + (j - CA) * (16 / (int)sizeof(T)));
            else if (j < CA + 2 * CX) cp_async16(&r_q[tok][(j - CA - CX) * (16 / (int)sizeof(T))], q + vec + (j - CA - CX) * (16 / (int)sizeof(T)));
            else cp_async16(&r_v[tok][(j - CA - 2 * CX) * (16 / (int)sizeof(T))], v + vec + (j - CA - 2 * CX) * (16 / (int)sizeof(T)));
        }
        if (t < gfirst) cp_async4b(&r_b[t], beta + (size_t)(n * n_tok + t) * H + h);
        asm volatile("cp.async.commit_group;" ::: "memory");
    };

    ptx::grid_dep_wait();      // (launched before the preceding kernel has ended)
    ptx::grid_dep_launch();
    int item = blockIdx.x;
    if (item < n_items) fetch(item);
    for (; item < n_items; item += gridDim.x) {
        const int n = item / H, h = item - n * H;
        float* Sp = state_of(item);
        float4 x[16];
        asm volatile("cp.async.wait_group 0;" ::: "memory");
#pragma unroll
        for (int m = 0; m < 16; ++m) x[m] = s_next[m * 256 + t];   // (each thread reads back its own copies)
        __syncthreads();   // the raw vectors were copied by other threads; the previous item's vectors are no longer read
        auto vec_of = [&](int tt) { return ((size_t)(n * n_tok + tt) * H + h) * kD; };
        for (int g0 = 0; g0 < n_tok; g0 += GT) {
            const int gn = (n_tok - g0) < GT ? (n_tok - g0) : GT;
            {   // thread (half, c): channel c of tokens half, half + 2, ...
                const int c = t & (kD - 1), half = t >> 7;
                if (g0 == 0) {   // from the prefetched raw vectors
#pragma unroll
                    for (int j = 0; j < GT / 2; ++j) {
                        const int tok = half + 2 * j;
                        if (tok < gn) {
                            const float kk = to_f<T>(r_k[tok][c]), bb = r_b[tok];
                            s_a[tok][at(c)] = expf(r_a[tok][c]);
                            s_k[tok][at(c)] = kk;
                            s_q[tok][at(c)] = to_f<T>(r_q[tok][c]);
                            s_bk[tok][at(c)] = bb * kk;
                            s_v[tok][c] = to_f<T>(r_v[tok][c]);
                            if (c == 0) s_b[tok] = bb;
                        }
                    }
                } else {         // later groups of a long call: straight from global memory, loads first
                    __syncthreads();   // the previous group's vectors are no longer read
                    float la[GT / 2], kk[GT / 2], qq[GT / 2], vv[GT / 2], bb[GT / 2];
#pragma unroll
                    for (int j = 0; j < GT / 2; ++j) {
                        const int tok = half + 2 * j;
                        if (tok < gn) {
                            const size_t vec = vec_of(g0 + tok) + c;
                            la[j] = log_alpha[vec];
                            kk[j] = to_f<T>(k[vec]);
                            qq[j] = to_f<T>(q[vec]);
                            vv[j] = to_f<T>(v[vec]);
                            bb[j] = beta[(size_t)(n * n_tok + g0 + tok) * H + h];
                        }
                    }
#pragma unroll
                    for (int j = 0; j < GT / 2; ++j) {
                        const int tok = half + 2 * j;
                        if (tok < gn) {
                            s_a[tok][at(c)] = expf(la[j]);
                            s_k[tok][at(c)] = kk[j];
                            s_q[tok][at(c)] = qq[j];
                            s_bk[tok][at(c)] = bb[j] * kk[j];
                            s_v[tok][c] = vv[j];
                            if (c == 0) s_b[tok] = bb[j];
                        }
                    }
                }
            }
            __syncthreads();
            // the raw buffers and the state buffer are free: the next item's data may stream in
            if (g0 == 0 && item + (int)gridDim.x < n_items) fetch(item + gridDim.x);
            if (warp < gn) {   // q.k of token `warp` (4 channels per lane, butterfly reduce)
                float qk = 0.f;
#pragma unroll
                for (int i = 0; i < 4; ++i) qk += s_q[warp][at(lane * 4 + i)] * s_k[warp][at(lane * 4 + i)];
#pragma unroll
                for (int ofs = 16; ofs > 0; ofs >>= 1) qk += __shfl_xor_sync(0xffffffffu, qk, ofs);
                if (lane == 0) s_qk[warp] = qk;
            }
            __syncthreads();
            for (int tok = 0; tok < gn; ++tok) {
                float4 p = make_float4(0.f, 0.f, 0.f, 0.f), s = p;
#pragma unroll
                for (int m = 0; m < 16; m += 4) {
                    const float4 ea = *reinterpret_cast<const float4*>(&s_a[tok][rg * L::kRow + m]);
                    const float4 ek = *reinterpret_cast<const float4*>(&s_k[tok][rg * L::kRow + m]);
                    const float4 eq = *reinterpret_cast<const float4*>(&s_q[tok][rg * L::kRow + m]);
                    mul4(x[m], ea.x);     fma4(p, ek.x, x[m]);     fma4(s, eq.x, x[m]);
                    mul4(x[m + 1], ea.y); fma4(p, ek.y, x[m + 1]); fma4(s, eq.y, x[m + 1]);
                    mul4(x[m + 2], ea.z); fma4(p, ek.z, x[m + 2]); fma4(s, eq.z, x[m + 2]);
                    mul4(x[m + 3], ea.w); fma4(p, ek.w, x[m + 3]); fma4(s, eq.w, x[m + 3]);
                    asm volatile("" ::: "memory");   // keeps the loads of later rows from being hoisted (registers)
                }
                // The eight row groups of a column group (lanes that differ in bits 2..4, fixed order), by halves: bit 2
                // keeps the sums of p or of s, bits 3 and 4 one column of the four; then every lane fetches p's.
                const bool b2 = lane & 4, b3 = lane & 8, b4 = lane & 16;
                float4 y = b2 ? s : p, w = b2 ? p : s;
                y.x += __shfl_xor_sync(0xffffffffu, w.x, 4); y.y += __shfl_xor_sync(0xffffffffu, w.y, 4);
                y.z += __shfl_xor_sync(0xffffffffu, w.z, 4); y.w += __shfl_xor_sync(0xffffffffu, w.w, 4);
                float2 y2 = b3 ? make_float2(y.z, y.w) : make_float2(y.x, y.y);
                const float2 w2 = b3 ? make_float2(y.x, y.y) : make_float2(y.z, y.w);
                y2.x += __shfl_xor_sync(0xffffffffu, w2.x, 8); y2.y += __shfl_xor_sync(0xffffffffu, w2.y, 8);
                const float sum = (b4 ? y2.y : y2.x) + __shfl_xor_sync(0xffffffffu, b4 ? y2.x : y2.y, 16);
                const float4 vv = *reinterpret_cast<const float4*>(&s_v[tok][col]);
                const float4 r = make_float4(vv.x - __shfl_sync(0xffffffffu, sum, cg), vv.y - __shfl_sync(0xffffffffu, sum, cg + 16),
                                             vv.z - __shfl_sync(0xffffffffu, sum, cg + 8), vv.w - __shfl_sync(0xffffffffu, sum, cg + 24));
                if (b2) {
                    const float c = s_b[tok] * s_qk[tok];
                    const float rr = b3 ? (b4 ? r.w : r.z) : (b4 ? r.y : r.x);
                    o[vec_of(g0 + tok) + col + (b3 ? 2 : 0) + (b4 ? 1 : 0)] = from_f<T>(scale * (sum + c * rr));
                }
#pragma unroll
                for (int m = 0; m < 16; m += 4) {
                    const float4 eb = *reinterpret_cast<const float4*>(&s_bk[tok][rg * L::kRow + m]);
                    fma4(x[m], eb.x, r); fma4(x[m + 1], eb.y, r); fma4(x[m + 2], eb.z, r); fma4(x[m + 3], eb.w, r);
                    asm volatile("" ::: "memory");
                }
            }
        }
#pragma unroll
        for (int m = 0; m < 16; ++m) st_stream(Sp + (size_t)(rg + 8 * m) * kD, x[m]);
    }
}

}  // namespace

kda_status_t sm_count(int* n_sm)
{
    DeviceLock lk;
    if (!lk.st) return lk.rc;
    if (lk.st->n_sm == 0) {
        int dev = 0;
        KDA_CUDA_TRY(cudaGetDevice(&dev));
        KDA_CUDA_TRY(cudaDeviceGetAttribute(&lk.st->n_sm, cudaDevAttrMultiProcessorCount, dev));
    }
    *n_sm = lk.st->n_sm;
    return KDA_OK;
}
namespace {
template <typename T, bool kLayer>
kda_status_t launch_decode_t(const void* q, const void* k, const void* v, const float* log_alpha, const float* beta,
                             float* S, const int32_t* slot, void* o, int n_seqs, int H, float scale,
                             const DecodeLayer& lay, cudaStream_t st)
{
    ProfScope ps(PROF_DECODE, st);
    int nc = kD;
    if (!kLayer) {
        int n_sm = 0;
        if (const kda_status_t rc = sm_count(&n_sm)) return rc;
        nc = decode_cols((int64_t)n_seqs * H, n_sm);
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)((size_t)n_seqs * H * (kD / nc)));
    cfg.blockDim = dim3(256);
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    auto kern = nc == kD ? kda_decode_kernel<T, kLayer, kD> : kda_decode_kernel<T, kLayer, kLayer ? kD : 64>;
    KDA_CUDA_TRY(cudaLaunchKernelEx(&cfg, kern, (const T*)q, (const T*)k, (const T*)v, log_alpha, beta, S, slot, (T*)o, H,
                                    scale, lay));
    count_launch();
    return KDA_OK;
}
}  // namespace

kda_status_t launch_decode(const void* q, const void* k, const void* v, const float* log_alpha,
                           const float* beta, float* S, const int32_t* slot, void* o, int n_seqs,
                           int H, float scale, kda_dtype_t dt, cudaStream_t st)
{
    if (n_seqs == 0) return KDA_OK;
    if (dt == KDA_BF16)
        return launch_decode_t<__nv_bfloat16, false>(q, k, v, log_alpha, beta, S, slot, o, n_seqs, H, scale, DecodeLayer(), st);
    return launch_decode_t<float, false>(q, k, v, log_alpha, beta, S, slot, o, n_seqs, H, scale, DecodeLayer(), st);
}

kda_status_t launch_layer_decode(const void* q_c, const void* k_c, const void* v, const void* g_a,
                                 const float* b_pre, const void* g_o, const float* A_log, const float* dt_bias,
                                 const float* rms_weight, float l2_eps, float rms_eps, float* S,
                                 const int32_t* slot, void* y, int n_seqs, int H, float scale, cudaStream_t st)
{
    if (n_seqs == 0) return KDA_OK;
    DecodeLayer lay;
    lay.A_log = A_log; lay.dt_bias = dt_bias; lay.g_o = g_o; lay.rms_weight = rms_weight;
    lay.l2_eps = l2_eps; lay.rms_eps = rms_eps;
    return launch_decode_t<__nv_bfloat16, true>(q_c, k_c, v, reinterpret_cast<const float*>(g_a), b_pre, S, slot, y, n_seqs,
                                                H, scale, lay, st);
}

kda_status_t launch_decode_multi(const void* q, const void* k, const void* v, const float* log_alpha,
                                 const float* beta, float* S, const int32_t* slot, void* o, int n_seqs,
                                 int n_tok, int H, float scale, kda_dtype_t dt, cudaStream_t st)
{
    if (n_seqs == 0 || n_tok == 0) return KDA_OK;
    int n_sm = 0;
    {
        DeviceLock lk;
        if (!lk.st) return lk.rc;
        if (!lk.st->attr_done[6]) {
            KDA_CUDA_TRY(cudaFuncSetAttribute(kda_decode_multi_kernel<__nv_bfloat16>,
                                              cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              MultiSmem<__nv_bfloat16>::kTotal));
            KDA_CUDA_TRY(cudaFuncSetAttribute(kda_decode_multi_kernel<float>,
                                              cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              MultiSmem<float>::kTotal));
            lk.st->attr_done[6] = true;
        }
        if (lk.st->n_sm == 0) {
            int dev = 0;
            KDA_CUDA_TRY(cudaGetDevice(&dev));
            KDA_CUDA_TRY(cudaDeviceGetAttribute(&lk.st->n_sm, cudaDevAttrMultiProcessorCount, dev));
        }
        n_sm = lk.st->n_sm;
    }
    const int n_items = n_seqs * H;
    const unsigned grid = (unsigned)(n_items < 2 * n_sm ? n_items : 2 * n_sm);   // persistent, two CTAs per SM
    ProfScope ps(PROF_DECODE, st);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(256);
    cfg.dynamicSmemBytes = dt == KDA_BF16 ? MultiSmem<__nv_bfloat16>::kTotal : MultiSmem<float>::kTotal;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (dt == KDA_BF16) {
        using T = __nv_bfloat16;
        KDA_CUDA_TRY(cudaLaunchKernelEx(&cfg, kda_decode_multi_kernel<T>, (const T*)q, (const T*)k, (const T*)v, log_alpha,
                                        beta, S, slot, (T*)o, H, n_tok, scale, n_items));
    } else {
        KDA_CUDA_TRY(cudaLaunchKernelEx(&cfg, kda_decode_multi_kernel<float>, (const float*)q, (const float*)k,
                                        (const float*)v, log_alpha, beta, S, slot, (float*)o, H, n_tok, scale, n_items));
    }
    count_launch();
    KDA_CUDA_TRY(cudaGetLastError());
    return KDA_OK;
}

}  // namespace kda
