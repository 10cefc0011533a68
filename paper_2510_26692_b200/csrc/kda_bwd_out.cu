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
// T=4096, H=32: warp-level tf32 products 784 us, 473 in this form.
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
// fp32 vectors (floats from O_VEC): beta[64] em[128] dbeta[8][64] sGC[4][128] colsum[2][64] seg[4][128], then barriers
constexpr int V_BETA = 0, V_EM = 64, V_DB = 192, V_GC = 704, V_CS = 1216, V_SEG = 1344, V_BAR = 1856;
constexpr uint32_t kSmem = O_VEC + V_BAR * 4 + 64 + 1024;     // + alignment slack
static_assert(4 * 64 * LR * 4 <= O_VEC, "the staged accumulators fit over the images");
static_assert(kSmem <= 232448, "fits the shared memory of one SM");
constexpr uint32_t C_P2 = 0, C_P4 = 128, C_P1 = 192, C_P6 = 256, C_P3 = 384;   // TMEM columns (P1: 192-319, read before P6)

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
    float* sBeta = vec + V_BETA; float* sDb = vec + V_DB; float* sEm = vec + V_EM; float* sGC = vec + V_GC;
    float* sCs = vec + V_CS; float* sSeg = vec + V_SEG;
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
    const int ra = t & 63, ca = (t >> 6) * 8;        // rf matrices of 64 rows: columns ca + 64 j
    const int rs = t & 127, cs = (t >> 7) * 8;       // and of 128 rows: columns cs + 32 j
    auto tok_off = [&](int r) { return ((size_t)(loc.tok0 + r) * a.H + h) * kD; };

    // ---- P1: dV -----------------------------------------------------------------------------------------
    Raw8<float> xs[4], rr[2];     // S now, Lam later; r
    {
        Raw8<float> xt, xx[2];
        const int r = t >> 3, x = (t & 7) * 8;
        ldraw(xt, tile + bt::T + r * 64 + x);
#pragma unroll
        for (int j = 0; j < 2; ++j) ldraw_rf(xx[j], tile + bt::X, 64, ra, ca + 64 * j);
#pragma unroll
        for (int j = 0; j < 2; ++j) ldraw_rf(rr[j], tile + bt::R, 64, ra, ca + 64 * j);
        const float b = r < loc.len ? a.beta[(size_t)(loc.tok0 + r) * a.H + h] : 0.f;
        const float em = tile[bt::EM + (t & 127)];
#pragma unroll
        for (int j = 0; j < 4; ++j) ldraw_rf(xs[j], tile + bt::S, 128, rs, cs + 32 * j);
        float v[8], u[8];
        to_f(xt, v);
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] *= b;
        put8<64, 1>(sm + O_RA, r, x, v);
        if (x == 0) sBeta[r] = b;
        if (t < 128) sEm[t] = em;
        float s = 0.f;      // share of r_j . dX_j
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            to_f(xx[j], v);
            to_f(rr[j], u);
            put8<64, 2>(sm + O_DX, ra, ca + 64 * j, v);
#pragma unroll
            for (int e = 0; e < 8; ++e) s = fmaf(v[e], u[e], s);
        }
        sDb[t] = s;         // [8][64]
    }
    Raw8<float> lam[4];
    Raw8<T> dd[2];
#pragma unroll
    for (int j = 0; j < 4; ++j) ldraw_rf(lam[j], tile + bt::L, 128, rs, cs + 32 * j);
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
    const uint32_t mnA = ptx::kIdescAMajorMN, mnB = ptx::kIdescBMajorMN;
    if (w == 0) {
        mma6<4>(tm + C_P1, mn_major<64, 1>(sm + O_RA), mn_major<64, 2>(sm + O_DX), ptx::umma_idesc_bf16(128, 128) | mnA | mnB, false);
        ptx::umma_commit(&bar[0]);
    }
    // meanwhile: e^(G_m) S, and its dot products with Lam
    {
        const float em = sEm[rs];
        float s = 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            float v[8], l[8];
            to_f(xs[j], v);
            to_f(lam[j], l);
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                s = fmaf(v[e], l[e], s);
                v[e] *= em;
            }
            put8<128, 2>(sm + O_RB, rs, cs + 32 * j, v);
        }
        sGC[t] = s * em * em;      // [4][128]; (G_m = G_C / 2)
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
    for (int j = 0; j < 2; ++j) {
        float v[8];
        to_f(dd[j], v);
        put8<128, 2>(sm + O_RA, row0 + 32 * j, c8, v);
    }
    publish();

    // ---- P2, then P4 and the first half of P3 ---------------------------------------------------------------
    if (w == 0) {
        mma6<8>(tm + C_P2, k_major<128, 2>(sm + O_RA), k_major<128, 2>(sm + O_RB), ptx::umma_idesc_bf16(128, 128), false);
        ptx::umma_commit(&bar[1]);
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
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        float v[8];
        to_f(rr[j], v);
        put8<64, 2>(sm + O_RB, ra, ca + 64 * j, v);
    }
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        float v[8];
        to_f(lam[j], v);
        put8<128, 1>(sm + O_LAM0, rs, cs + 32 * j, v);
    }
    publish();
    if (w == 0) {
        mma6<8>(tm + C_P4, k_major<128, 2>(sm + O_RA), k_major<64, 2>(sm + O_RB), ptx::umma_idesc_bf16(128, 64), false);
        ptx::umma_commit(&bar[2]);
        mma6<4>(tm + C_P3, k_major<64, 2>(sm + O_RB), k_major<128, 1>(sm + O_LAM0), ptx::umma_idesc_bf16(128, 128), false);
    }
    wait(2);
#pragma unroll
    for (int j = 2; j < 4; ++j) {
        float v[8];
        to_f(lam[j], v);
        put8<128, 1>(sm + O_LAM1, rs, cs + 32 * j - 64, v);
    }
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
    if (w == 0) {
        mma6<4>(tm + C_P3, k_major<64, 2>(sm + O_RB + 8192), k_major<128, 1>(sm + O_LAM1), ptx::umma_idesc_bf16(128, 128), true);
        ptx::umma_commit(&bar[3]);
    }
    if (t < loc.len) {
        float s = sCs[t] + sCs[64 + t];
#pragma unroll
        for (int j = 0; j < 8; ++j) s += sDb[j * 64 + t];
        a.db[(size_t)(loc.tok0 + t) * a.H + h] = s;
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
    if (w == 0) {
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
    const float ec = sEm[c];          // e^(G_C - G_m): G_m = G_C / 2
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
    float dG[16], run = 0.f, gsum = 0.f;
#pragma unroll
    for (int i = 15; i >= 0; --i) {
        const int r = seg * 16 + i;
        const size_t off = tok_off(r) + c;
        const bool in = r < loc.len;
        const float f1 = gv[i], f2 = reciprocal(f1);
        const float dq = a.scale * f1 * stage[r * LR + c];
        const float p3 = ec * f2 * stage[(192 + r) * LR + c];       // e^(G_C - G) (beta r Lam^T)
        const float dk1 = f1 * stage[(64 + r) * LR + c], dk2 = fmaf(f2, stage[(128 + r) * LR + c], p3);
        if (in) {
            a.dq[off] = dq;
            a.dk[off] = dk1 + dk2;
        }
        gsum = fmaf(kv[i], p3, gsum);
        run += fmaf(qv[i], dq, kv[i] * (dk1 - dk2));
        dG[i] = run;
    }
    // d G_C: all segments' sums of K~ dK~ and e^(G_C) rowsum(S Lam)
    float* sSum = stage + 256 * LR;      // [4][128], behind the staged accumulators
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
