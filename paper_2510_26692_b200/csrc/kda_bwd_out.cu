// Gradients stage of the chunkwise backward pass (equations in kda_bwd_chunk.cu): one CTA per (chunk, head),
// every product on tcgen05 with split operands (kda_split3.cuh), accumulators in TMEM.
//
// The products of a tile and where their operand images live (RA, RB: 96 KB each; rows x columns):
//   P1  dV  = (beta T')^T dX              T' 64x64, dX 64x128 in RA
//   P2  e^(G_m) [dO ; -dV] S^T            [dO ; -dV] 128x128 in RA, e^(G_m) S 128x128 in RB
//   P4  [dO ; -dV] r^T                    r 64x128 in RB (over S)
//   P3  r Lam^T                           Lam's column halves: in RB beside r, then in RA
//   P5  P2 += [dP ; dB] K_                [dP ; dB] 128x64 and K_ 64x128 in RA
//   P6  [dP ; dB]^T [Q ; K^]              [Q ; K^] 128x128 in RB
// While the tensor core works on one product the threads fetch and split the operands of the next.
//
// T=4096, H=32: warp-level tf32 products (the form before) 784 us; this form: see launch_bwd_out.
#include "kda_bwd.cuh"
#include "kda_split3.cuh"

namespace kda {
namespace {

using namespace split3;
constexpr int kT = 512;
constexpr int LR = 132;
constexpr uint32_t O_RA = 0, O_RB = 98304, O_VEC = 196608;
constexpr uint32_t O_DX = O_RA + 3 * 8192;                    // dX beside T'
constexpr uint32_t O_LAM0 = O_RB + 3 * 16384;                 // Lam, v columns 0-63, beside r
constexpr uint32_t O_LAM1 = O_RA;                             // Lam, v columns 64-127; then K_
constexpr uint32_t O_DPB = O_RA + 3 * 16384;                  // [dP ; dB]
// fp32 vectors (floats from O_VEC): beta[64] dbeta[64] gm[128] sGC[128] colsum[2][64] seg[4][128], then barriers
constexpr int V_BETA = 0, V_DB = 64, V_GM = 128, V_GC = 256, V_CS = 384, V_SEG = 512, V_BAR = 1024;
constexpr uint32_t kSmem = O_VEC + V_BAR * 4 + 64 + 1024;     // + alignment slack
static_assert(4 * 64 * LR * 4 <= O_VEC, "the staged accumulators fit over the images");
static_assert(kSmem <= 232448, "fits the shared memory of one SM");
constexpr uint32_t C_P2 = 0, C_P4 = 128, C_P1 = 192, C_P6 = 256, C_P3 = 384;   // TMEM columns (P1: 192-319, read before P6)

__device__ __forceinline__ void ld8(const float* p, float (&x)[8]) {
    const float4 a = *reinterpret_cast<const float4*>(p), b = *reinterpret_cast<const float4*>(p + 4);
    x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w; x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
}
__device__ __forceinline__ void ld8(const __nv_bfloat16* p, float (&x)[8]) {
    const uint4 a = *reinterpret_cast<const uint4*>(p);
    const uint32_t w[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) { x[2 * e] = __uint_as_float(w[e] << 16); x[2 * e + 1] = __uint_as_float(w[e] & 0xffff0000u); }
}

template <typename T>
__global__ void __launch_bounds__(kT, 1) kda_bwd_out(BwdChunkArgs a)
{
    extern __shared__ uint8_t smem_raw[];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    const int h = blockIdx.y;
    if (a.seq_heads[h]) return;
    uint8_t* sm = smem_raw + ((1024u - (ptx::smem_u32(smem_raw) & 1023u)) & 1023u);
    float* vec = reinterpret_cast<float*>(sm + O_VEC);
    float* sBeta = vec + V_BETA; float* sDb = vec + V_DB; float* sGm = vec + V_GM; float* sGC = vec + V_GC;
    float* sCs = vec + V_CS; float* sSeg = vec + V_SEG;
    uint64_t* bar = reinterpret_cast<uint64_t*>(vec + V_BAR);   // one per group of MMAs, each used once
    uint32_t* slot = reinterpret_cast<uint32_t*>(bar + 6);
    const BwdLoc loc = bwd_locate(a, blockIdx.x);
    const float* tile = a.tiles + ((size_t)blockIdx.x * a.H + h) * bt::kFloats;

    if (w == 0) {
        ptx::tmem_alloc(slot, 512);
        ptx::tmem_relinquish();
    }
    if (t == 32) {
#pragma unroll
        for (int i = 0; i < 6; ++i) ptx::mbar_init(&bar[i], 1);
        ptx::fence_mbar_init();
    }
    bool ok = true;
    auto wait = [&](int i) {
        if (ok) ok = ptx::mbar_wait(&bar[i], 0, a.wait_limit_ns);
        __syncwarp();
        ptx::tc_fence_after();
    };
    auto publish = [&]() {     // shared-memory images written by all threads -> visible to the MMA
        ptx::fence_async_smem();
        ptx::tc_fence_before();
        __syncthreads();
        ptx::tc_fence_after();
    };
    // unit u of a matrix with 128 columns: row u >> 4, columns 8 (u & 15) .. + 7
    const int c8 = (t & 15) * 8, row0 = t >> 4;      // rows row0 + 32 j
    auto tok_off = [&](int r) { return ((size_t)(loc.tok0 + r) * a.H + h) * kD; };

    // ---- P1: dV -----------------------------------------------------------------------------------------
    float xs[4][8];     // S now, Lam later
#pragma unroll
    for (int j = 0; j < 4; ++j) ld8(tile + bt::S + (row0 + 32 * j) * kD + c8, xs[j]);
    {
        const int r = t >> 3, x = (t & 7) * 8;
        float v[8];
        ld8(tile + bt::T + r * 64 + x, v);
        const float b = r < loc.len ? a.beta[(size_t)(loc.tok0 + r) * a.H + h] : 0.f;
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] *= b;
        put8<64, 1>(sm + O_RA, r, x, v);
        if (x == 0) sBeta[r] = b;
    }
    float rr[2][8];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int r = row0 + 32 * j;
        float v[8];
        ld8(tile + bt::X + r * kD + c8, v);
        ld8(tile + bt::R + r * kD + c8, rr[j]);
        put8<64, 2>(sm + O_DX, r, c8, v);
        float s = 0.f;      // r_j . dX_j
#pragma unroll
        for (int e = 0; e < 8; ++e) s = fmaf(v[e], rr[j][e], s);
#pragma unroll
        for (int o = 1; o < 16; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((t & 15) == 0) sDb[r] = s;
    }
    if (t < 128) sGm[t] = 0.5f * tile[bt::G + 63 * kD + t];
    publish();
    const uint32_t tm = *slot;
    const uint32_t mnA = ptx::kIdescAMajorMN, mnB = ptx::kIdescBMajorMN;
    if (t == 0) {
        mma6<4>(tm + C_P1, mn_major<64, 1>(sm + O_RA), mn_major<64, 2>(sm + O_DX), ptx::umma_idesc_bf16(128, 128) | mnA | mnB, false);
        ptx::umma_commit(&bar[0]);
    }
    // meanwhile: e^(G_m) S, and its dot products with Lam
    float dd[2][8];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int r = row0 + 32 * j;
#pragma unroll
        for (int e = 0; e < 8; ++e) dd[j][e] = 0.f;
        if (r < loc.len && a.d_o) ld8(reinterpret_cast<const T*>(a.d_o) + tok_off(r) + c8, dd[j]);
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        const int r = row0 + 32 * j;
        const float em = expf(sGm[r]);
        float v[8], l[8];
        ld8(tile + bt::L + r * kD + c8, l);
        float s = 0.f;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            s = fmaf(xs[j][e], l[e], s);
            v[e] = em * xs[j][e];
            xs[j][e] = l[e];
        }
        put8<128, 2>(sm + O_RB, r, c8, v);
#pragma unroll
        for (int o = 1; o < 16; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((t & 15) == 0) sGC[r] = s * tile[bt::GC + r];
    }
    wait(0);
    // dV: rows = TMEM lanes 0-63 (warps of quadrants 0 and 1), 32 columns each
    const int quad = w & 3, cg = (w >> 2) * 32;
    const uint32_t tq = tm + ((uint32_t)(quad * 32) << 16);
    if (quad < 2) {
        const int i = quad * 32 + lane;
        uint32_t y[32];
        ptx::tmem_ld_32x32b_x32(tq + C_P1 + cg, y);
        ptx::tmem_ld_wait();
        if (i < loc.len) {
            float* p = a.dv + tok_off(i) + cg;
#pragma unroll
            for (int e = 0; e < 32; e += 4)
                *reinterpret_cast<uint4*>(p + e) = make_uint4(y[e], y[e + 1], y[e + 2], y[e + 3]);
        }
#pragma unroll
        for (int q8 = 0; q8 < 4; ++q8) {
            float v[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] = -__uint_as_float(y[8 * q8 + e]);
            put8<128, 2>(sm + O_RA, 64 + i, cg + 8 * q8, v);
        }
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) put8<128, 2>(sm + O_RA, row0 + 32 * j, c8, dd[j]);
    publish();

    // ---- P2, then P4 and the first half of P3 ---------------------------------------------------------------
    if (t == 0) {
        mma6<8>(tm + C_P2, k_major<128, 2>(sm + O_RA), k_major<128, 2>(sm + O_RB), ptx::umma_idesc_bf16(128, 128), false);
        ptx::umma_commit(&bar[1]);
    }
    wait(1);
#pragma unroll
    for (int j = 0; j < 2; ++j) put8<64, 2>(sm + O_RB, row0 + 32 * j, c8, rr[j]);
    if (c8 < 64)
#pragma unroll
        for (int j = 0; j < 4; ++j) put8<128, 1>(sm + O_LAM0, row0 + 32 * j, c8, xs[j]);
    publish();
    if (t == 0) {
        mma6<8>(tm + C_P4, k_major<128, 2>(sm + O_RA), k_major<64, 2>(sm + O_RB), ptx::umma_idesc_bf16(128, 64), false);
        ptx::umma_commit(&bar[2]);
        mma6<4>(tm + C_P3, k_major<64, 2>(sm + O_RB), k_major<128, 1>(sm + O_LAM0), ptx::umma_idesc_bf16(128, 128), false);
    }
    // the gated operands' inputs, requested while the tensor core works
    float kk[2][8], qq[2][8], gg[2][8];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int r = row0 + 32 * j;
#pragma unroll
        for (int e = 0; e < 8; ++e) kk[j][e] = qq[j][e] = 0.f;
        if (r < loc.len) {
            ld8(reinterpret_cast<const T*>(a.k) + tok_off(r) + c8, kk[j]);
            ld8(reinterpret_cast<const T*>(a.q) + tok_off(r) + c8, qq[j]);
        }
        ld8(tile + bt::G + r * kD + c8, gg[j]);
    }
    wait(2);
    if (c8 >= 64)
#pragma unroll
        for (int j = 0; j < 4; ++j) put8<128, 1>(sm + O_LAM1, row0 + 32 * j, c8 - 64, xs[j]);
    {   // masked and scaled Gram matrices; columns j0 .. j0 + 15 of row lane + 32 quad of [dP ; dB]
        const int R = quad * 32 + lane, i = R & 63, j0 = (w >> 2) * 16;
        const bool isB = quad >= 2;
        uint32_t y[16];
        ptx::tmem_ld_32x32b_x16(tq + C_P4 + j0, y);
        float bb[16];
        if (isB) {
#pragma unroll
            for (int e = 0; e < 16; e += 4) {
                const float4 v = *reinterpret_cast<const float4*>(tile + bt::B + i * 64 + j0 + e);
                bb[e] = v.x; bb[e + 1] = v.y; bb[e + 2] = v.z; bb[e + 3] = v.w;
            }
        }
        ptx::tmem_ld_wait();
        float v[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            v[e] = j0 + e + (isB ? 1 : 0) <= i ? __uint_as_float(y[e]) : 0.f;
            if (isB) bb[e] *= v[e];              // B_ij (-dV_i . r_j)
            v[e] *= sBeta[j0 + e];
        }
        float lo[8], hi[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) { lo[e] = v[e]; hi[e] = v[8 + e]; }
        put8<128, 1>(sm + O_DPB, R, j0, lo);
        put8<128, 1>(sm + O_DPB, R, j0 + 8, hi);
        if (isB) {   // column sums over the warp's 32 rows: 16 values over 32 lanes
#pragma unroll
            for (int s = 8; s >= 1; s >>= 1) {
                const bool up = (lane & s) != 0;
#pragma unroll
                for (int e = 0; e < s; ++e) {
                    const float send = up ? bb[e] : bb[e + s], keep = up ? bb[e + s] : bb[e];
                    bb[e] = keep + __shfl_xor_sync(0xffffffffu, send, s);
                }
            }
            bb[0] += __shfl_xor_sync(0xffffffffu, bb[0], 16);
            if (lane < 16) sCs[(quad - 2) * 64 + j0 + lane] = bb[0];
        }
    }
    publish();
    if (t == 0) {
        mma6<4>(tm + C_P3, k_major<64, 2>(sm + O_RB + 8192), k_major<128, 1>(sm + O_LAM1), ptx::umma_idesc_bf16(128, 128), true);
        ptx::umma_commit(&bar[3]);
    }
    if (t < loc.len) a.db[(size_t)(loc.tok0 + t) * a.H + h] = sDb[t] + (sCs[t] + sCs[64 + t]);
    // gates in place of G: exp(G - G_m), exp(G_m - G)
    float e1[2][8];
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const float x = gg[j][e] - sGm[c8 + e];
            e1[j][e] = expf(x);
            gg[j][e] = kk[j][e] * expf(-x);          // K_
            kk[j][e] *= e1[j][e];                    // K^
            qq[j][e] *= a.scale * e1[j][e];          // Q
        }
    wait(3);

    // ---- P5, P6 -------------------------------------------------------------------------------------------
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int r = row0 + 32 * j;
        put8<64, 2>(sm + O_LAM1, r, c8, gg[j]);
        put8<128, 2>(sm + O_RB, r, c8, qq[j]);
        put8<128, 2>(sm + O_RB, 64 + r, c8, kk[j]);
    }
    publish();
    if (t == 0) {
        mma6<4>(tm + C_P2, k_major<128, 1>(sm + O_DPB), mn_major<64, 2>(sm + O_LAM1), ptx::umma_idesc_bf16(128, 128) | mnB, true);
        mma6<8>(tm + C_P6, mn_major<128, 1>(sm + O_DPB), mn_major<128, 2>(sm + O_RB), ptx::umma_idesc_bf16(128, 128) | mnA | mnB, false);
        ptx::umma_commit(&bar[4]);
    }
    // accumulators to shared memory: [0] dQ, [1] dK^, [2] dK_, [3] beta r Lam^T, rows = tokens.  P3 first: it is complete.
    float* stage = reinterpret_cast<float*>(sm);
    uint32_t y3[32];
    if (quad < 2) {
        ptx::tmem_ld_32x32b_x32(tq + C_P3 + cg, y3);
        ptx::tmem_ld_wait();
    }
    // the column pass's inputs: thread = channel c of 16 consecutive tokens
    const int c = t & 127, seg = t >> 7;
    const float gm = sGm[c];
    wait(4);
    {
        uint32_t y[32];
        ptx::tmem_ld_32x32b_x32(tq + C_P2 + cg, y);
        ptx::tmem_ld_wait();
        float* p = stage + (quad * 32 + lane) * LR + cg;
#pragma unroll
        for (int e = 0; e < 32; e += 4) *reinterpret_cast<uint4*>(p + e) = make_uint4(y[e], y[e + 1], y[e + 2], y[e + 3]);
    }
    if (quad < 2) {
        const int i = quad * 32 + lane;
        uint32_t y[32];
        ptx::tmem_ld_32x32b_x32(tq + C_P6 + cg, y);
        ptx::tmem_ld_wait();
        float* p = stage + (128 + i) * LR + cg;
        const float b = sBeta[i];
#pragma unroll
        for (int e = 0; e < 32; e += 4) {
            *reinterpret_cast<uint4*>(p + e) = make_uint4(y[e], y[e + 1], y[e + 2], y[e + 3]);
            *reinterpret_cast<float4*>(p + 64 * LR + e) =
                make_float4(b * __uint_as_float(y3[e]), b * __uint_as_float(y3[e + 1]), b * __uint_as_float(y3[e + 2]),
                            b * __uint_as_float(y3[e + 3]));
        }
    }
    ptx::tc_fence_before();
    __syncthreads();
    const T* kp = reinterpret_cast<const T*>(a.k);
    const T* qp = reinterpret_cast<const T*>(a.q);
    const float ec = expf(gm);        // e^(G_C - G_m): G_m = G_C / 2
    float dG[16], run = 0.f, gsum = 0.f;
#pragma unroll
    for (int i = 15; i >= 0; --i) {
        const int r = seg * 16 + i;
        const size_t off = tok_off(r) + c;
        const bool in = r < loc.len;
        const float x = tile[bt::G + r * kD + c] - gm;
        const float kv = in ? (float)kp[off] : 0.f, qv = in ? (float)qp[off] : 0.f;
        const float f1 = expf(x), f2 = expf(-x);
        const float dq = a.scale * f1 * stage[r * LR + c];
        const float p3 = ec * f2 * stage[(192 + r) * LR + c];       // e^(G_C - G) (beta r Lam^T)
        const float dk1 = f1 * stage[(64 + r) * LR + c], dk2 = fmaf(f2, stage[(128 + r) * LR + c], p3);
        if (in) {
            a.dq[off] = dq;
            a.dk[off] = dk1 + dk2;
        }
        gsum = fmaf(kv, p3, gsum);
        run += fmaf(qv, dq, kv * (dk1 - dk2));
        dG[i] = run;
    }
    // d G_C: all segments' sums of K~ dK~ and e^(G_C) rowsum(S Lam)
    float* sSum = stage + 256 * LR;      // [4][128], behind the staged accumulators
    sSeg[seg * 128 + c] = run;
    sSum[seg * 128 + c] = gsum;
    __syncthreads();
    float base = sGC[c] + ((sSum[c] + sSum[128 + c]) + (sSum[256 + c] + sSum[384 + c]));
    for (int s = 3; s > seg; --s) base += sSeg[s * 128 + c];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const int r = seg * 16 + i;
        if (r < loc.len) a.dg[tok_off(r) + c] = dG[i] + base;
    }
    if (!ok && atomicCAS(&a.hdr->status, 0, (int)KDA_ERR_TIMEOUT) == 0) a.hdr->where = 30;
    __syncthreads();
    if (w == 0) ptx::tmem_dealloc(tm, 512);
}

}  // namespace

kda_status_t launch_bwd_out(const BwdChunkArgs& a, kda_dtype_t dt, cudaStream_t st)
{
    {
        DeviceLock lk;
        if (!lk.st) return lk.rc;
        if (!lk.st->attr_done[14]) {
            KDA_CUDA_TRY(cudaFuncSetAttribute(kda_bwd_out<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem));
            KDA_CUDA_TRY(cudaFuncSetAttribute(kda_bwd_out<__nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem));
            lk.st->attr_done[14] = true;
        }
    }
    const dim3 grid((unsigned)a.n_chunks, (unsigned)a.H);
    ProfScope ps(PROF_INTRA, st);
    if (dt == KDA_BF16) kda_bwd_out<__nv_bfloat16><<<grid, kT, kSmem, st>>>(a);
    else kda_bwd_out<float><<<grid, kT, kSmem, st>>>(a);
    count_launch();
    KDA_CUDA_TRY(cudaGetLastError());
    return KDA_OK;
}

}  // namespace kda
