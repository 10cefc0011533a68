// Gradients stage of the chunkwise backward pass (equations in kda_bwd_chunk.cu): one CTA per (chunk, head),
// every product on tcgen05 with split operands (kda_split3.cuh), accumulators in TMEM.
//
// The products of a tile (M x N x K) and where their operands live: D and X are regions of shared memory of 96 KB each, A
// the 192 TMEM columns of an A operand.
//   P1  dV = (beta T')^T dX                 T' 64x64 and dX^T 128x64 in X
//   P2  e^(G_m) S [dO ; -dV]^T              S in A, [dO ; -dV] 128x128 in D
//   P4  [dO ; -dV] r^T                      r^T 128x64 in X
//   P3  Lam r^T                             Lam in A
//   P5  P2 += K_^T [dP ; dB]^T              [dP ; dB] 128x64 and K_ 64x128 in X
//   P6  [Q ; K^]^T [dP ; dB]                [Q ; K^] 128x128 in D
// P2, P3, P5 and P6 have the channels in the TMEM lanes, so that the pass over the columns (a thread per channel) reads them
// there.  Operands in shared memory are what these products are bound by: a product of 128 x 128 x 16 reads 8 KB of it
// in the 64 clocks that it takes, all there is, and with A in TMEM half of that.
//
// T=4096, H=32: warp-level tf32 products 784 us; all operands in shared memory and accumulators staged there 418; 341 in
// this form.
#include "kda_bwd.cuh"
#include "kda_split3.cuh"

namespace kda {
namespace {

using namespace split3;
constexpr int kT = 512;
constexpr int kIssue = 15;                                    // the warp that issues the MMAs
constexpr uint32_t O_D = 0, O_X = 98304, O_VEC = 196608;
constexpr uint32_t O_T = O_X, O_DX = O_X + 24576;             // T', dX
constexpr uint32_t O_R = O_X, O_DPB = O_X + 49152;            // r, later K_; [dP ; dB]
// fp32 vectors (floats from O_VEC): beta[64] dbeta[4][64] sGC[4][128] colsum[2][64] seg[4][128] sum[4][128], then barriers
constexpr int V_BETA = 0, V_DB = 64, V_GC = 320, V_CS = 832, V_SEG = 960, V_SUM = 1472, V_BAR = 1984;
constexpr uint32_t kSmem = O_VEC + V_BAR * 4 + 64 + 1024;     // + alignment slack
static_assert(kSmem <= 232448, "fits the shared memory of one SM");
// TMEM columns; P1 (128) lies where P3 and P6 come to lie
constexpr uint32_t C_A = 0, kAParts = 64, C_P2 = 192, C_P4 = 320, C_P1 = 384, C_P3 = 384, C_P6 = 448;

__device__ __forceinline__ float ldv(const float* p, bool in) {
    float x = 0.f;
    if (in) asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(x) : "l"(p));
    return x;
}
__device__ __forceinline__ float ldv(const __nv_bfloat16* p, bool in) {
    unsigned short x = 0;
    if (in) asm volatile("ld.global.nc.u16 %0, [%1];" : "=h"(x) : "l"(p));
    return __uint_as_float((uint32_t)x << 16);
}

// sums of 16 values over the warp; lane l gets number l % 16 in s[0] (each exchange halves the values a lane carries)
__device__ __forceinline__ void lane_sums(float (&s)[16], int lane) {
#pragma unroll
    for (int n = 8; n >= 1; n >>= 1) {
        const bool up = (lane & n) != 0;
#pragma unroll
        for (int e = 0; e < n; ++e) {
            const float send = up ? s[e] : s[e + n], keep = up ? s[e + n] : s[e];
            s[e] = keep + __shfl_xor_sync(0xffffffffu, send, n);
        }
    }
    s[0] += __shfl_xor_sync(0xffffffffu, s[0], 16);
}

template <typename T>
__global__ void __launch_bounds__(kT, 1) kda_bwd_out(BwdChunkArgs a)
{
    extern __shared__ uint8_t smem_raw[];
    const int t = threadIdx.x, lane = t & 31, w = ptx::warp_uniform(t >> 5);
    int64_t chunk; int h;
    bwd_tile(a, blockIdx.x, chunk, h);
    if (a.seq_heads[h]) return;
    uint8_t* sm = smem_raw + ((1024u - (ptx::smem_u32(smem_raw) & 1023u)) & 1023u);
    float* vec = reinterpret_cast<float*>(sm + O_VEC);
    float* sBeta = vec + V_BETA; float* sDb = vec + V_DB; float* sGC = vec + V_GC;
    float* sCs = vec + V_CS; float* sSeg = vec + V_SEG; float* sSum = vec + V_SUM;
    uint64_t* bar = reinterpret_cast<uint64_t*>(vec + V_BAR);   // one per group of MMAs, each used once
    uint32_t* slot = reinterpret_cast<uint32_t*>(bar + 6);
    const BwdLoc loc = bwd_locate(a, chunk);
    const float* tile = a.tiles + (size_t)blockIdx.x * bt::kFloats;

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
    const int c8 = (t & 15) * 8, row0 = t >> 4;      // token tensors: rows row0 + 32 j
    const int rs = t & 127, cs = (t >> 7) * 32;      // matrices of 128 rows (TMEM lane rs): columns cs + 8 j, or ct + 8 j of 64
    const int ct = (t >> 7) * 16;
    auto tok_off = [&](int r) { return ((size_t)(loc.tok0 + r) * a.H + h) * kD; };

    // ---- P1: dV -----------------------------------------------------------------------------------------
    Raw8<float> xs[4], rr[2];     // S, r
    const float em = tile[bt::EM + rs];      // of row rs of S, and of channel rs in the pass over the columns
    {
        Raw8<float> xt, xx[2];
        const int r = t >> 3, x = (t & 7) * 8;
        ldraw(xt, tile + bt::T + r * 64 + x);
#pragma unroll
        for (int j = 0; j < 2; ++j) ldraw_rf(xx[j], tile + bt::X, 128, rs, ct + 8 * j);
#pragma unroll
        for (int j = 0; j < 2; ++j) ldraw_rf(rr[j], tile + bt::R, 128, rs, ct + 8 * j);
        const float b = r < loc.len ? a.beta[(size_t)(loc.tok0 + r) * a.H + h] : 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) ldraw_sf(xs[j], tile + bt::S, rs, cs + 8 * j);
        float v[8], u[8];
        to_f(xt, v);
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] *= b;
        put8<64, 1>(sm + O_T, r, x, v);
        if (x == 0) sBeta[r] = b;
        float s[16];      // shares of r_j . dX_j, j = ct ..: column rs of both
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            to_f(xx[j], v);
            to_f(rr[j], u);
            put8<128, 1>(sm + O_DX, rs, ct + 8 * j, v);
#pragma unroll
            for (int e = 0; e < 8; ++e) s[8 * j + e] = v[e] * u[e];
        }
        lane_sums(s, lane);
        if (lane < 16) sDb[(w & 3) * 64 + ct + lane] = s[0];
    }
    Raw8<float> lam[4];
    Raw8<T> dd[2];
#pragma unroll
    for (int j = 0; j < 4; ++j) ldraw_sf(lam[j], tile + bt::L, rs, cs + 8 * j);
#pragma unroll
    for (int j = 0; j < 2; ++j)
        ldraw(dd[j], static_cast<const T*>(a.d_o) + tok_off(row0 + 32 * j) + c8, row0 + 32 * j < loc.len && a.d_o);
    {   // see prefetch_l2
        int64_t ng; int nh;
        if (bwd_next(a, blockIdx.x, ng, nh)) {
            const float* nt = a.tiles + ((size_t)ng * a.H + nh) * bt::kFloats;
            if (t == kT - 32) prefetch_l2(nt + bt::R, 2 * 64 * kD * 4);
            if (t == kT - 64) prefetch_l2(nt + bt::S, (bt::kFloats - bt::S) * 4);
            prefetch_rows<kT, T, 3>(bwd_locate(a, ng), a.H, nh, t, {static_cast<const T*>(a.k), static_cast<const T*>(a.q), static_cast<const T*>(a.d_o)});
        }
    }
    publish();
    const uint32_t tm = (uint32_t)ptx::warp_uniform((int)*slot);
    const uint32_t mnA = ptx::kIdescAMajorMN, mnB = ptx::kIdescBMajorMN, id = ptx::umma_idesc_bf16(128, 128);
    const int quad = w & 3, seg = w >> 2;
    const uint32_t tq = tm + ((uint32_t)(quad * 32) << 16);
    if (w == kIssue) {
        mma6<4>(tm + C_P1, mn_major<64, 1>(sm + O_T, 0, true), k_major<128, 1>(sm + O_DX), id | mnA, false);
        ptx::umma_commit(&bar[0]);
    }
    // meanwhile: e^(G_m) S, and its dot products with Lam; dO
    {
        float s = 0.f;
        float2 x[16];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float v[8], l[8];
            to_f(xs[j], v);
            to_f(lam[j], l);
#pragma unroll
            for (int e = 0; e < 8; ++e) s = fmaf(v[e], l[e], s);
#pragma unroll
            for (int e = 0; e < 4; ++e) x[4 * j + e] = make_float2(v[2 * e] * em, v[2 * e + 1] * em);
        }
        put_tmem<kAParts>(tq + C_A + seg * 16, x);
        sGC[t] = s * em * em;      // [4][128]; (G_m = G_C / 2)
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        float v[8];
        to_f(dd[j], v);
        put8<128, 2>(sm + O_D, row0 + 32 * j, c8, v);
    }
    ptx::tmem_st_wait();
    wait(0);
    {   // dV: rows = TMEM lanes 0-63, repeated in lanes 64-127; 16 columns a thread.  r over T' and dX
        const int i = (quad & 1) * 32 + lane, c0 = seg * 32 + (quad >> 1) * 16;
        uint32_t y[16];
        ptx::tmem_ld_32x32b_x16(tq + C_P1 + c0, y);
        ptx::tmem_ld_wait();
        if (i < loc.len) {
            float* p = a.dv + tok_off(i) + c0;
#pragma unroll
            for (int e = 0; e < 16; e += 4)
                *reinterpret_cast<uint4*>(p + e) = make_uint4(y[e], y[e + 1], y[e + 2], y[e + 3]);
        }
        float v[8];
#pragma unroll
        for (int q8 = 0; q8 < 2; ++q8) {
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] = -__uint_as_float(y[8 * q8 + e]);
            put8<128, 2>(sm + O_D, 64 + i, c0 + 8 * q8, v);
        }
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            to_f(rr[j], v);
            put8<128, 1>(sm + O_R, rs, ct + 8 * j, v);
        }
    }
    publish();

    // ---- P2, P4 ---------------------------------------------------------------------------------------------
    if (w == kIssue) {
        mma6_ta<8, kAParts>(tm + C_P2, tm + C_A, k_major<128, 2>(sm + O_D), id, false);
        ptx::umma_commit(&bar[1]);
        mma6<8>(tm + C_P4, k_major<128, 2>(sm + O_D), mn_major<128, 1>(sm + O_R), ptx::umma_idesc_bf16(128, 64) | mnB, false);
        ptx::umma_commit(&bar[2]);
    }
    // the gated operands' inputs, requested while the tensor core works
    Raw8<T> kr[2], qr[2];
    Raw8<float> gr[2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int r = row0 + 32 * j;
        ldraw(kr[j], static_cast<const T*>(a.k) + tok_off(r) + c8, r < loc.len);
        ldraw(qr[j], static_cast<const T*>(a.q) + tok_off(r) + c8, r < loc.len);
        ldraw(gr[j], tile + bt::F + r * kD + c8);
    }
    wait(1);
    {   // Lam over S
        float2 x[16];
#pragma unroll
        for (int j = 0; j < 4; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) x[4 * j + e] = make_float2(__uint_as_float(lam[j].w[2 * e]), __uint_as_float(lam[j].w[2 * e + 1]));
        put_tmem<kAParts>(tq + C_A + seg * 16, x);
        ptx::tmem_st_wait();
    }
    publish();
    if (w == kIssue) {
        mma6_ta<8, kAParts>(tm + C_P3, tm + C_A, mn_major<128, 1>(sm + O_R), ptx::umma_idesc_bf16(128, 64) | mnB, false);
        ptx::umma_commit(&bar[3]);
    }
    wait(2);
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
            lane_sums(bb, lane);
            if (lane < 16) sCs[(quad - 2) * 64 + j0 + lane] = bb[0];
        }
    }
    // gated operands: exp(G - G_m), exp(G_m - G)
    float kk[2][8], qq[2][8], gg[2][8];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        to_f(kr[j], kk[j]);
        to_f(qr[j], qq[j]);
        to_f(gr[j], gg[j]);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const float f1 = gg[j][e];
            gg[j][e] = kk[j][e] * reciprocal(f1);     // K_
            kk[j][e] *= f1;                          // K^
            qq[j][e] *= a.scale * f1;                // Q
        }
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        const int r = row0 + 32 * j;
        put8<128, 2>(sm + O_D, r, c8, qq[j]);
        put8<128, 2>(sm + O_D, 64 + r, c8, kk[j]);
    }
    wait(3);              // r has been read: K_ over it
#pragma unroll
    for (int j = 0; j < 2; ++j) put8<64, 2>(sm + O_R, row0 + 32 * j, c8, gg[j]);
    publish();

    // ---- P5, P6 -------------------------------------------------------------------------------------------
    if (w == kIssue) {
        mma6<4>(tm + C_P2, mn_major<64, 2>(sm + O_R), k_major<128, 1>(sm + O_DPB), id | mnA, true);
        mma6<8>(tm + C_P6, mn_major<128, 2>(sm + O_D), mn_major<128, 1>(sm + O_DPB), ptx::umma_idesc_bf16(128, 64) | mnA | mnB, false);
        ptx::umma_commit(&bar[4]);
    }
    if (t < loc.len) {
        float s = sCs[t] + sCs[64 + t];
#pragma unroll
        for (int j = 0; j < 4; ++j) s += sDb[j * 64 + t];
        a.db[(size_t)(loc.tok0 + t) * a.H + h] = s;
    }
    // the column pass's inputs: thread = channel c of 16 consecutive tokens
    const int c = rs;
    const float ec = em;              // e^(G_C - G_m): G_m = G_C / 2
    const T* kp = static_cast<const T*>(a.k);
    const T* qp = static_cast<const T*>(a.q);
    float kv[16], qv[16], gv[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const int r = seg * 16 + i;
        const bool in = r < loc.len;
        kv[i] = ldv(kp + tok_off(r) + c, in);
        qv[i] = ldv(qp + tok_off(r) + c, in);
        gv[i] = ldv(tile + bt::F + r * kD + c, true);
    }
    wait(4);
    float dG[16], run = 0.f, gsum = 0.f;
#pragma unroll
    for (int half = 1; half >= 0; --half) {
        uint32_t yq[8], yk[8], y6[8], y3[8];      // dQ, dK^, dK_, Lam r^T before the gates
        const uint32_t at = tq + seg * 16 + half * 8;
        ptx::tmem_ld_32x32b_x8(at + C_P2, yq);
        ptx::tmem_ld_32x32b_x8(at + C_P2 + 64, yk);
        ptx::tmem_ld_32x32b_x8(at + C_P6, y6);
        ptx::tmem_ld_32x32b_x8(at + C_P3, y3);
        ptx::tmem_ld_wait();
#pragma unroll
        for (int x = 7; x >= 0; --x) {
            const int i = half * 8 + x, r = seg * 16 + i;
            const size_t off = tok_off(r) + c;
            const float f1 = gv[i], f2 = reciprocal(f1);
            const float dq = a.scale * f1 * __uint_as_float(yq[x]);
            const float p3 = ec * f2 * (sBeta[r] * __uint_as_float(y3[x]));       // e^(G_C - G) (beta r Lam^T)
            const float dk1 = f1 * __uint_as_float(yk[x]), dk2 = fmaf(f2, __uint_as_float(y6[x]), p3);
            if (r < loc.len) {
                a.dq[off] = dq;
                a.dk[off] = dk1 + dk2;
            }
            gsum = fmaf(kv[i], p3, gsum);
            run += fmaf(qv[i], dq, kv[i] * (dk1 - dk2));
            dG[i] = run;
        }
    }
    // d G_C: all segments' sums of K~ dK~ and e^(G_C) rowsum(S Lam)
    sSeg[seg * 128 + c] = run;
    sSum[seg * 128 + c] = gsum;
    __syncthreads();
    float base = ((sGC[c] + sGC[128 + c]) + (sGC[256 + c] + sGC[384 + c])) + ((sSum[c] + sSum[128 + c]) + (sSum[256 + c] + sSum[384 + c]));
    for (int s = 3; s > seg; --s) base += sSeg[s * 128 + c];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
        const int r = seg * 16 + i;
        if (r < loc.len) a.dg[tok_off(r) + c] = dG[i] + base;
    }
    if (!ok && atomicCAS(&a.hdr->status, 0, (int)KDA_ERR_TIMEOUT) == 0) a.hdr->where = 30;
    ptx::tc_fence_before();
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
    const dim3 grid((unsigned)(a.n_chunks * a.H));
    ProfScope ps(PROF_INTRA, st);
    if (dt == KDA_BF16) kda_bwd_out<__nv_bfloat16><<<grid, kT, kSmem, st>>>(a);
    else kda_bwd_out<float><<<grid, kT, kSmem, st>>>(a);
    count_launch();
    KDA_CUDA_TRY(cudaGetLastError());
    return KDA_OK;
}

}  // namespace kda
