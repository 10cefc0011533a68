// Gradients stage of the chunkwise backward pass (equations in kda_bwd_chunk.cu): a CTA per SM goes through the (chunk, head)
// tiles, every product on tcgen05 with split operands (kda_split3.cuh), accumulators in TMEM.
//
// The products of a tile (M x N x K) and where their operands live: D, r, P regions of shared memory, A the 192 TMEM
// columns of an A operand.
//   P1  dV = (beta T')^T dX                 T' 64x64 and dX^T 128x64
//   P2  e^(G_m) S [dO ; -dV]^T              S in A, [dO ; -dV] 128x128 in D
//   P4  [dO ; -dV] r^T                      r^T 128x64 in r
//   P3  Lam r^T                             Lam in A
//   P5  P2 += K_^T [dP ; dB]^T              [dP ; dB] 128x64 in P, K_^T 128x64 in D
//   P6  [Q ; K^]^T [dP ; dB]                [Q ; K^]^T 128x128 in A
// P2, P3, P5 and P6 have the channels in the TMEM lanes, so that the pass over the columns (a thread per channel) reads them
// there.  Operands in shared memory are what these products are bound by: a product of 128 x 128 x 16 reads 8 KB of it
// in the 64 clocks that it takes, all there is, and with A in TMEM half of that.
//
// Warps 0-15 compute, 16 issues the MMAs (a warp that also computed held up the others by the 1900 clocks that 48 MMAs
// take to issue), 17 loads: the fp32 matrices of the next tile land in the shared memory that is free during the pass over
// the columns.  No register to spare: a few spilled ones cost a tenth (beside 225 KB of shared memory the L1 holds none).
//
// T=4096, H=32: warp-level tf32 products 784 us; all operands in shared memory and accumulators staged there 418; a CTA a tile
// that loaded into registers 350; 295 in this form.
#include "kda_bwd.cuh"
#include "kda_split3.cuh"

namespace kda {
namespace {

using namespace split3;
constexpr int kT = 640, kCompute = 512;
constexpr int kRegs = 112, kRegsRest = 32;      // of a compute thread and of the others: 512 x 112 + 128 x 32 <= 640 x 96
// What lands there, and the images that come to lie over it once it has been read
constexpr uint32_t K = 1024;
constexpr uint32_t O_S = 0, O_XX = 64 * K, O_RR = 96 * K, O_TT = 128 * K, O_LL = 152 * K;      // S, X, R, T', Lam
constexpr uint32_t O_D = 0, O_DX = 64 * K, O_R = 96 * K, O_T = 128 * K, O_DPB = 152 * K, O_VEC = 216 * K;
// fp32 vectors (floats from O_VEC): beta[64] dbeta[4][64] sGC[4][128] colsum[2][64] seg[4][128] sum[4][128], those of the tile,
// then barriers
constexpr int V_BETA = 0, V_DB = 64, V_GC = 320, V_CS = 832, V_SEG = 960, V_SUM = 1472, V_TILE = 1984, V_BAR = V_TILE + bt::kVec;
constexpr uint32_t kSmem = O_VEC + V_BAR * 4 + 128 + 1024;    // + alignment slack
static_assert(kSmem <= 232448, "fits the shared memory of one SM");
static_assert(V_BAR % 2 == 0 && V_TILE % 4 == 0, "barriers and bulk copies are aligned");
// TMEM columns; P1 (128) lies where P3 and P6 come to lie
constexpr uint32_t C_A = 0, kAParts = 64, C_P2 = 192, C_P4 = 320, C_P1 = 384, C_P3 = 384, C_P6 = 448;

__device__ __forceinline__ float ldv(const float* p) {
    float x;
    asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(x) : "l"(p));
    return x;
}
// 16 tokens of one channel as they are stored, two bf16 a register once they have arrived (pack)
template <typename T> struct Column;
template <> struct Column<float> {
    float v[16];
    __device__ __forceinline__ void load(int i, const float* p, bool in) {
        v[i] = 0.f;
        if (in) v[i] = ldv(p);
    }
    __device__ __forceinline__ void pack() {}
    __device__ __forceinline__ void again() {}
    __device__ __forceinline__ float at(int i) const { return v[i]; }
};
template <> struct Column<__nv_bfloat16> {
    unsigned short u[16];
    uint32_t v[8];
    __device__ __forceinline__ void load(int i, const __nv_bfloat16* p, bool in) {
        u[i] = 0;
        if (in) asm volatile("ld.global.nc.u16 %0, [%1];" : "=h"(u[i]) : "l"(p));
    }
    __device__ __forceinline__ void pack() {
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] = (uint32_t)u[2 * e] | (uint32_t)u[2 * e + 1] << 16;
    }
    // what was unpacked is not kept from here on but unpacked again
    __device__ __forceinline__ void again() {
#pragma unroll
        for (int e = 0; e < 8; ++e) asm volatile("" : "+r"(v[e]));
    }
    __device__ __forceinline__ float at(int i) const { return __uint_as_float(i & 1 ? v[i >> 1] & 0xffff0000u : v[i >> 1] << 16); }
};

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
    uint8_t* sm = smem_raw + ((1024u - (ptx::smem_u32(smem_raw) & 1023u)) & 1023u);
    float* vec = reinterpret_cast<float*>(sm + O_VEC);
    float* sBeta = vec + V_BETA; float* sDb = vec + V_DB; float* sGC = vec + V_GC;
    float* sCs = vec + V_CS; float* sSeg = vec + V_SEG; float* sSum = vec + V_SUM;
    const float* sTile = vec + V_TILE;
    // a phase of each per tile: groups of MMAs complete, their operands written (16 warps), the tile's matrices landed
    uint64_t* bar = reinterpret_cast<uint64_t*>(vec + V_BAR);
    uint64_t* ready = bar + 5;
    uint64_t* landed = ready + 4;
    uint64_t* done = landed + 1;       // (once) all MMAs complete
    uint32_t* slot = reinterpret_cast<uint32_t*>(done + 1);
    if (w == kCompute / 32) {
        ptx::tmem_alloc(slot, 512);
        ptx::tmem_relinquish();
        if (lane == 0) {
#pragma unroll
            for (int i = 0; i < 11; ++i) ptx::mbar_init(&bar[i], i >= 5 && i < 9 ? kCompute / 32 : 1);
            ptx::fence_mbar_init();
        }
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tm = (uint32_t)ptx::warp_uniform((int)*slot);
    bool ok = true;
    uint32_t phase = 0;
    auto wait_on = [&](uint64_t* b) {
        if (ok) ok = ptx::mbar_wait(b, phase, a.wait_limit_ns);
        __syncwarp();
        ptx::tc_fence_after();
    };
    ptx::grid_dep_wait();      // (launched before the preceding kernel has ended)
    // tiles of this CTA: id, id + gridDim.x, ... without those of heads that are not in chunk form
    uint32_t id = blockIdx.x;      // (fewer than 2^31 tiles)
    int h = 0;
    int64_t chunk = 0;
    auto find = [&]() {
        for (; id < (uint32_t)(a.n_chunks * a.H); id += gridDim.x) {
            bwd_tile(a, id, chunk, h);
            if (!a.seq_heads[h]) return true;
        }
        return false;
    };
    if (w >= kCompute / 32) {
        ptx::reg_dec<kRegsRest>();
        const uint32_t mnA = ptx::kIdescAMajorMN, mnB = ptx::kIdescBMajorMN, id64 = ptx::umma_idesc_bf16(128, 64), id128 = ptx::umma_idesc_bf16(128, 128);
        if (w == kCompute / 32) {
            // ================= MMAs =================
            for (; find(); id += gridDim.x) {
                wait_on(&ready[0]);
                mma6<4>(tm + C_P1, mn_major<64, 1>(sm + O_T, 0, true), k_major<128, 1>(sm + O_DX), id128 | mnA, false);
                ptx::umma_commit(&bar[0]);
                wait_on(&ready[1]);
                mma6_ta<8, kAParts>(tm + C_P2, tm + C_A, k_major<128, 2>(sm + O_D), id128, false);
                ptx::umma_commit(&bar[1]);
                mma6<8>(tm + C_P4, k_major<128, 2>(sm + O_D), mn_major<128, 1>(sm + O_R), id64 | mnB, false);
                ptx::umma_commit(&bar[2]);
                wait_on(&ready[2]);
                mma6_ta<8, kAParts>(tm + C_P3, tm + C_A, mn_major<128, 1>(sm + O_R), id64 | mnB, false);
                ptx::umma_commit(&bar[3]);
                wait_on(&ready[3]);
                mma6<4>(tm + C_P2, k_major<128, 1>(sm + O_D), k_major<128, 1>(sm + O_DPB), id128, true);
                mma6_ta<8, kAParts>(tm + C_P6, tm + C_A, mn_major<128, 1>(sm + O_DPB), id64 | mnB, false);
                ptx::umma_commit(&bar[4]);
                phase ^= 1u;
            }
            ptx::umma_commit(done);        // before the TMEM goes away, also where a wait has run out
            if (!ptx::mbar_wait(done, 0, a.wait_limit_ns)) ok = false;
            __syncwarp();
        } else if (w == kCompute / 32 + 1) {
            // ================= loads =================
            while (find()) {
                if (lane == 0) {
                    const float* tile = a.tiles + (size_t)id * bt::kFloats;
                    ptx::mbar_expect_tx(landed, (2 * bt::kState + 2 * 64 * kD + 64 * 64 + bt::kVec) * 4);
                    ptx::bulk_g2s(sm + O_TT, tile + bt::T, 64 * 64 * 4, landed);
                    ptx::bulk_g2s(sm + O_VEC + V_TILE * 4, tile + bt::GC, bt::kVec * 4, landed);
                    ptx::bulk_g2s(sm + O_XX, tile + bt::X, 64 * kD * 4, landed);
                    ptx::bulk_g2s(sm + O_RR, tile + bt::R, 64 * kD * 4, landed);
                    ptx::bulk_g2s(sm + O_S, tile + bt::S, bt::kState * 4, landed);
                    ptx::bulk_g2s(sm + O_LL, tile + bt::L, bt::kState * 4, landed);
                }
                __syncwarp();
                {   // see prefetch_l2
                    int64_t ng; int nh;
                    if (bwd_next(a, id, ng, nh)) {
                        const float* nt = a.tiles + ((size_t)ng * a.H + nh) * bt::kFloats;
                        if (lane == 0) prefetch_l2(nt + bt::R, 2 * 64 * kD * 4);
                        if (lane == 0) prefetch_l2(nt + bt::S, (bt::kFloats - bt::S) * 4);
                        prefetch_rows<32, T, 3>(bwd_locate(a, ng), a.H, nh, lane, {static_cast<const T*>(a.k), static_cast<const T*>(a.q), static_cast<const T*>(a.d_o)});
                    }
                }
                id += gridDim.x;
                wait_on(&bar[4]);      // no operand is needed any more
                if (!ok) ptx::mbar_wait(landed, phase, a.wait_limit_ns);     // (nothing may be in flight when the CTA leaves)
                phase ^= 1u;
            }
        }
        if (lane == 0 && !ok && atomicCAS(&a.hdr->status, 0, (int)KDA_ERR_TIMEOUT) == 0) a.hdr->where = 30;
        __syncwarp();
        __syncthreads();
        ptx::tc_fence_after();
        if (w == kCompute / 32) ptx::tmem_dealloc(tm, 512);
        return;
    }
    ptx::reg_inc<kRegs>();
    auto barrier = [&]() { ptx::named_bar_sync(1, kCompute); };
    auto publish = [&](int i) {     // shared-memory images and TMEM operands written by this warp -> visible to the MMA
        ptx::fence_async_smem();
        ptx::tc_fence_before();
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(&ready[i]);
    };
    const int c8 = (t & 15) * 8, row0 = t >> 4;      // token tensors: rows row0 + 32 j, columns c8 ..
    const int rs = t & 127, cs = (t >> 7) * 32;      // matrices of 128 rows (TMEM lane rs): columns cs + 8 j, or ct + 8 j of 64
    const int ct = (t >> 7) * 16, quad = w & 3, seg = w >> 2;
    const uint32_t tq = tm + ((uint32_t)(quad * 32) << 16);
    // eight values of a matrix that has landed
    auto lds = [&](float (&x)[8], uint32_t at, int p0, int p1) {
        const float4 u = *reinterpret_cast<const float4*>(sm + at + p0 * 4), v = *reinterpret_cast<const float4*>(sm + at + p1 * 4);
        x[0] = u.x; x[1] = u.y; x[2] = u.z; x[3] = u.w; x[4] = v.x; x[5] = v.y; x[6] = v.z; x[7] = v.w;
    };
    for (; find(); id += gridDim.x) {
        const BwdLoc loc = bwd_locate(a, chunk);
        const float* tile = a.tiles + (size_t)id * bt::kFloats;
        auto tok_off = [&](int r) { return ((size_t)(loc.tok0 + r) * a.H + h) * kD; };
        Raw8<T> dd[2];
#pragma unroll
        for (int j = 0; j < 2; ++j)
            ldraw(dd[j], static_cast<const T*>(a.d_o) + tok_off(row0 + 32 * j) + c8, row0 + 32 * j < loc.len && a.d_o);

        // ---- P1: dV -------------------------------------------------------------------------------------
        wait_on(landed);
        const float em = sTile[bt::EM - bt::GC + rs];      // of row rs of S, and of channel rs in the pass over the columns
        float rr[2][8];
        {
            float v[8], xx[2][8], s[16];      // s: shares of r_j . dX_j, j = ct ..: column rs of both
            const int r = t >> 3, x = (t & 7) * 8;
            lds(v, O_TT, r * 64 + x, r * 64 + x + 4);
            const float b = sTile[bt::BE - bt::GC + r];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                lds(xx[j], O_XX, rf(128, rs, ct + 8 * j), rf(128, rs, ct + 8 * j + 4));
                lds(rr[j], O_RR, rf(128, rs, ct + 8 * j), rf(128, rs, ct + 8 * j + 4));
            }
            if (x == 0) sBeta[r] = b;
            barrier();        // T', X and R have been read: images over them
#pragma unroll
            for (int e = 0; e < 8; ++e) v[e] *= b;
            put8<64, 1>(sm + O_T, r, x, v);
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                put8<128, 1>(sm + O_DX, rs, ct + 8 * j, xx[j]);
#pragma unroll
                for (int e = 0; e < 8; ++e) s[8 * j + e] = xx[j][e] * rr[j][e];
            }
            publish(0);
            lane_sums(s, lane);
            if (lane < 16) sDb[quad * 64 + ct + lane] = s[0];
        }
        // meanwhile: e^(G_m) S, and its dot products with Lam
        {
            float s = 0.f;
#pragma unroll
            for (int jj = 0; jj < 4; jj += 2) {
                float2 x[8];
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    float v[8], l[8];
                    lds(v, O_S, sf(rs, cs + 8 * (jj + j)), sf(rs, cs + 8 * (jj + j) + 4));
                    lds(l, O_LL, sf(rs, cs + 8 * (jj + j)), sf(rs, cs + 8 * (jj + j) + 4));
#pragma unroll
                    for (int e = 0; e < 8; ++e) s = fmaf(v[e], l[e], s);
#pragma unroll
                    for (int e = 0; e < 4; ++e) x[4 * j + e] = make_float2(v[2 * e] * em, v[2 * e + 1] * em);
                }
                put_tmem<kAParts>(tq + C_A + seg * 16 + jj * 4, x);
            }
            sGC[t] = s * em * em;      // [4][128]; (G_m = G_C / 2)
            ptx::tmem_st_wait();
        }
        wait_on(&bar[0]);
        barrier();            // S has been read: [dO ; -dV] over it
        {   // dV: rows = TMEM lanes 0-63, repeated in lanes 64-127; 16 columns a thread
            const int i = (quad & 1) * 32 + lane, c0 = seg * 32 + (quad >> 1) * 16;
            uint32_t y[16];
            ptx::tmem_ld_32x32b_x16(tq + C_P1 + c0, y);
            float v[8];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                to_f(dd[j], v);
                put8<128, 2>(sm + O_D, row0 + 32 * j, c8, v);
                put8<128, 1>(sm + O_R, rs, ct + 8 * j, rr[j]);
            }
            ptx::tmem_ld_wait();
            if (i < loc.len) {
                float* p = a.dv + tok_off(i) + c0;
#pragma unroll
                for (int e = 0; e < 16; e += 4)
                    *reinterpret_cast<uint4*>(p + e) = make_uint4(y[e], y[e + 1], y[e + 2], y[e + 3]);
            }
#pragma unroll
            for (int q8 = 0; q8 < 2; ++q8) {
#pragma unroll
                for (int e = 0; e < 8; ++e) v[e] = -__uint_as_float(y[8 * q8 + e]);
                put8<128, 2>(sm + O_D, 64 + i, c0 + 8 * q8, v);
            }
        }
        publish(1);

        // ---- P2, P4 -------------------------------------------------------------------------------------
        // the gated operands' inputs, requested while the tensor core works: thread = channel c of 16 consecutive tokens
        const int c = rs;
        Column<T> kv, qv;
        float gv[16];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const int r = seg * 16 + i;
            const size_t off = tok_off(r) + c;
            kv.load(i, static_cast<const T*>(a.k) + off, r < loc.len);
            qv.load(i, static_cast<const T*>(a.q) + off, r < loc.len);
            gv[i] = ldv(tile + bt::F + r * kD + c);
        }
        kv.pack(); qv.pack();      // (they arrive before the product does)
        wait_on(&bar[1]);
        {   // Lam over S
#pragma unroll
            for (int jj = 0; jj < 4; jj += 2) {
                float2 x[8];
#pragma unroll
                for (int j = 0; j < 2; ++j) {
                    float l[8];
                    lds(l, O_LL, sf(rs, cs + 8 * (jj + j)), sf(rs, cs + 8 * (jj + j) + 4));
#pragma unroll
                    for (int e = 0; e < 4; ++e) x[4 * j + e] = make_float2(l[2 * e], l[2 * e + 1]);
                }
                put_tmem<kAParts>(tq + C_A + seg * 16 + jj * 4, x);
            }
            ptx::tmem_st_wait();
        }
        publish(2);
        float bb[16];         // of B, for the rows of dB
        const int R = quad * 32 + lane, j0 = seg * 16;
        if (quad >= 2) {
#pragma unroll
            for (int e = 0; e < 16; e += 4) {
                const float4 v = *reinterpret_cast<const float4*>(tile + bt::B + (R & 63) * 64 + j0 + e);
                bb[e] = v.x; bb[e + 1] = v.y; bb[e + 2] = v.z; bb[e + 3] = v.w;
            }
        }
        wait_on(&bar[2]);
        barrier();            // Lam has been read: [dP ; dB] over it
        {   // masked and scaled Gram matrices; columns j0 .. j0 + 15 of row lane + 32 quad of [dP ; dB]
            const int i = R & 63;
            const bool isB = quad >= 2;
            uint32_t y[16];
            ptx::tmem_ld_32x32b_x16(tq + C_P4 + j0, y);
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
        kv.again();
        // gated operands: K_ over [dO ; -dV], [Q ; K^] over Lam
#pragma unroll
        for (int q8 = 0; q8 < 2; ++q8) {
            float x[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) x[e] = kv.at(8 * q8 + e) * reciprocal(gv[8 * q8 + e]);
            put8<128, 1>(sm + O_D, c, seg * 16 + 8 * q8, x);
        }
        kv.again(); qv.again();
        wait_on(&bar[3]);
        {
            float2 x[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) x[e] = make_float2(qv.at(2 * e) * (a.scale * gv[2 * e]), qv.at(2 * e + 1) * (a.scale * gv[2 * e + 1]));
            put_tmem<kAParts>(tq + C_A + seg * 8, x);
#pragma unroll
            for (int e = 0; e < 8; ++e) x[e] = make_float2(kv.at(2 * e) * gv[2 * e], kv.at(2 * e + 1) * gv[2 * e + 1]);
            put_tmem<kAParts>(tq + C_A + 32 + seg * 8, x);
            ptx::tmem_st_wait();
        }
        publish(3);
        barrier();            // (column sums)

        // ---- P5, P6 -----------------------------------------------------------------------------------------
        if (t < loc.len) {
            float s = sCs[t] + sCs[64 + t];
#pragma unroll
            for (int j = 0; j < 4; ++j) s += sDb[j * 64 + t];
            a.db[(size_t)(loc.tok0 + t) * a.H + h] = s;
        }
        const float ec = em;              // e^(G_C - G_m): G_m = G_C / 2
        kv.again(); qv.again();
        wait_on(&bar[4]);
        float dG[16], run = 0.f, gsum = 0.f;
#pragma unroll
        for (int q = 3; q >= 0; --q) {
            uint32_t yq[4], yk[4], y6[4], y3[4];      // dQ, dK^, dK_, Lam r^T before the gates
            const uint32_t at = tq + seg * 16 + q * 4;
            ptx::tmem_ld_32x32b_x4(at + C_P2, yq);
            ptx::tmem_ld_32x32b_x4(at + C_P2 + 64, yk);
            ptx::tmem_ld_32x32b_x4(at + C_P6, y6);
            ptx::tmem_ld_32x32b_x4(at + C_P3, y3);
            ptx::tmem_ld_wait();
#pragma unroll
            for (int x = 3; x >= 0; --x) {
                const int i = q * 4 + x, r = seg * 16 + i;
                const size_t off = tok_off(r) + c;
                const float f1 = gv[i], f2 = reciprocal(f1);
                const float dq = a.scale * f1 * __uint_as_float(yq[x]);
                const float p3 = ec * f2 * (sBeta[r] * __uint_as_float(y3[x]));       // e^(G_C - G) (beta r Lam^T)
                const float dk1 = f1 * __uint_as_float(yk[x]), dk2 = fmaf(f2, __uint_as_float(y6[x]), p3);
                if (r < loc.len) {
                    a.dq[off] = dq;
                    a.dk[off] = dk1 + dk2;
                }
                gsum = fmaf(kv.at(i), p3, gsum);
                run += fmaf(qv.at(i), dq, kv.at(i) * (dk1 - dk2));
                dG[i] = run;
            }
        }
        // d G_C: all segments' sums of K~ dK~ and e^(G_C) rowsum(S Lam)
        sSeg[seg * 128 + c] = run;
        sSum[seg * 128 + c] = gsum;
        barrier();
        float base = ((sGC[c] + sGC[128 + c]) + (sGC[256 + c] + sGC[384 + c])) + ((sSum[c] + sSum[128 + c]) + (sSum[256 + c] + sSum[384 + c]));
        for (int s = 3; s > seg; --s) base += sSeg[s * 128 + c];
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const int r = seg * 16 + i;
            if (r < loc.len) a.dg[tok_off(r) + c] = dG[i] + base;
        }
        phase ^= 1u;
    }
    ptx::grid_dep_launch();
    if (!ok && atomicCAS(&a.hdr->status, 0, (int)KDA_ERR_TIMEOUT) == 0) a.hdr->where = 30;
    ptx::tc_fence_before();
    __syncthreads();
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
    const int64_t tiles = a.n_chunks * a.H;
    const unsigned grid = (unsigned)(tiles < a.n_sm ? tiles : a.n_sm);
    ProfScope ps(PROF_INTRA, st);
    KDA_CUDA_TRY(launch_dependent(dt == KDA_BF16 ? kda_bwd_out<__nv_bfloat16> : kda_bwd_out<float>, dim3(grid), kT, kSmem, st, a));
    count_launch();
    return KDA_OK;
}

}  // namespace kda
