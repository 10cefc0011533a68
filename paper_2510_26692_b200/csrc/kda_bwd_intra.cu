// First stage of the chunkwise backward pass (equations in kda_bwd_chunk.cu): everything of a (chunk, head) tile
// that depends on neither state.  Products on tcgen05 with split operands
// (kda_split3.cuh); the 64 x 64 inverse (16 x 16 blocks by fp32 substitution, joined by split tf32 products, kda_mma3.cuh) runs
// beside the two products that do not need it.
//
//   A   [K^ ; Q] K_^T        -> B (masked), P (masked)
//   C1  dO^T Q               -> N            C2  dO^T P -> X
//   D1  K^^T T'^T            -> W'^T         D2  V^T T'^T -> U'^T
// (the 64-row matrices as the N side: 128 x 64 x 16 takes the tensor core half of 128 x 128 x 16).  dO and V that are stored
// in bf16 are operands as they are.  Shared memory: RQ 96 KB [K^ ; Q], later the W'^T image; RK 48 KB K_, then V;
// L, T' fp32; RP 24 KB P, then T'; dO in a place of its own (bf16) or in RK before V.
//
// T=4096, H=32: 470 us with warp-level tf32 products; with all operands split and 64-row products on 128 rows 271; 223
// in this form.
#include "kda_bwd.cuh"
#include "kda_mma3.cuh"
#include "kda_split3.cuh"

namespace kda {
namespace {

using namespace split3;
constexpr int kT = 512;
constexpr int kIssue = 15;              // the warp that issues the MMAs (it has no part in the inverse)
constexpr int LM = 68;
constexpr uint32_t O_RQ = 0, O_RK = 98304, O_RP = O_RK + 49152, O_L = O_RP + 24576, O_T = O_L + 64 * LM * 4,
                   O_G = O_RP,                       // e^(G - G_m) [64][132] fp32 before P, L and T' exist
                   O_DO = O_T + 64 * LM * 4, O_VEC = O_DO + 16384;
static_assert(O_G + 64 * 132 * 4 <= O_DO, "G fits where P, L and T' come to lie");
constexpr int V_BETA = 0, V_SEG = 64, V_BAR = 1088;     // floats: beta, segment sums [2][4][128], barriers
constexpr uint32_t kSmem = O_VEC + V_BAR * 4 + 64 + 1024;
static_assert(kSmem <= 232448, "fits the shared memory of one SM");
constexpr uint32_t C_N = 0, C_X = 128, C_A = 192, C_W = 256, C_U = 320;   // TMEM columns

template <typename T>
__global__ void __launch_bounds__(kT, 1) kda_bwd_intra(BwdChunkArgs a)
{
    extern __shared__ uint8_t smem_raw[];
    const int t = threadIdx.x, lane = t & 31, w = ptx::warp_uniform(t >> 5);
    uint8_t* sm = smem_raw + ((1024u - (ptx::smem_u32(smem_raw) & 1023u)) & 1023u);
    float* vec = reinterpret_cast<float*>(sm + O_VEC);
    float* sBeta = vec + V_BETA; float* sSeg = vec + V_SEG;
    uint64_t* bar = reinterpret_cast<uint64_t*>(vec + V_BAR);   // one per group of MMAs, a phase per tile
    uint64_t* done = bar + 4;      // all MMAs complete, where a wait has run out
    uint32_t* slot = reinterpret_cast<uint32_t*>(done + 1);

    ptx::grid_dep_wait();      // (launched before the preceding kernel has ended)
    // bf16 rows: a CTA per SM goes through the tiles, and the inputs of the next are requested as soon as
    // their registers are free (4096 x 32 heads 285 -> 271 us; all of them during the last products: 230, now 223).  fp32 rows take twice the registers, and
    // spilled (67 -> 77 us on six packed sequences): a CTA per tile.
    constexpr bool kExact = sizeof(T) == 2, kLoop = kExact;
    const int64_t n_tiles = a.n_chunks * a.H;
    int64_t id = blockIdx.x;
    int h;
    BwdLoc loc = {};
    const int c = t & 127, seg = t >> 7;          // the decay: thread = channel c of 16 consecutive tokens
    const int c8 = (t & 15) * 8, row0 = t >> 4;   // token tensors by units of eight columns: rows row0 + 32 j, columns c8 ..
    float G[16], b_next = 0.f;
    Raw8<T> kr[2], qr[2], dr[2], vr[2];
    auto tok_off = [&](int r) { return ((size_t)(loc.tok0 + r) * a.H + h) * kD; };
    auto request = [&]() {
        int64_t chunk;
        bwd_tile(a, id, chunk, h);
        loc = bwd_locate(a, chunk);
        if (t < 64) b_next = t < loc.len ? a.beta[(size_t)(loc.tok0 + t) * a.H + h] : 0.f;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
            const int r = seg * 16 + i;
            G[i] = 0.f;
            if (r < loc.len) asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(G[i]) : "l"(a.log_alpha + tok_off(r) + c));
        }
    };
    auto request_rows = [&]() {
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int r = row0 + 32 * j;
            const size_t off = tok_off(r) + c8;
            const bool in = r < loc.len;
            ldraw(kr[j], static_cast<const T*>(a.k) + off, in);
            ldraw(qr[j], static_cast<const T*>(a.q) + off, in);
            ldraw(dr[j], static_cast<const T*>(a.d_o) + off, in && a.d_o);
        }
    };
    auto request_v = [&]() {
#pragma unroll
        for (int j = 0; j < 2; ++j) ldraw(vr[j], static_cast<const T*>(a.v) + tok_off(row0 + 32 * j) + c8, row0 + 32 * j < loc.len);
    };
    request();
    request_rows();
    request_v();
    if (w == 0) {
        ptx::tmem_alloc(slot, 512);
        ptx::tmem_relinquish();
    }
    if (t == 32) {
#pragma unroll
        for (int i = 0; i < 5; ++i) ptx::mbar_init(&bar[i], 1);
        ptx::fence_mbar_init();
    }
    bool ok = true;
    uint32_t phase = 0;
    auto wait = [&](int i) {
        if (ok) ok = ptx::mbar_wait(&bar[i], phase, a.wait_limit_ns);
        __syncwarp();
        ptx::tc_fence_after();
    };
    // a unit of a bf16 matrix as the first split of its image
    auto put_exact = [&](uint8_t* img, int r, int col, const Raw8<T>& x) {
        *reinterpret_cast<uint4*>(img + (col >> 6) * 8192 + ptx::sw128_off((uint32_t)r, (uint32_t)(col & 63))) = make_uint4(x.w[0], x.w[1], x.w[2], x.w[3]);
    };
    auto publish = [&]() {     // shared-memory images written by all threads -> visible to the MMA and the TMA engine
        ptx::fence_async_smem();
        ptx::tc_fence_before();
        __syncthreads();
        ptx::tc_fence_after();
    };
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tm = (uint32_t)ptx::warp_uniform((int)*slot);
    const uint32_t mnA = ptx::kIdescAMajorMN, mnB = ptx::kIdescBMajorMN;
    constexpr int kCopy = 64;      // the thread that issues the bulk copies

    while (true) {
        float* tile = a.tiles + (size_t)id * bt::kFloats;
        const int head = h, marked = *reinterpret_cast<volatile int*>(a.seq_heads + h);    // (by a tile before this one)
        if (t < 64) sBeta[t] = b_next;
        {
            int64_t ng; int nh;
            if (bwd_next(a, id, ng, nh)) {   // see prefetch_l2
                const BwdLoc nl = bwd_locate(a, ng);
                prefetch_rows<kT, float, 1>(nl, a.H, nh, t, {a.log_alpha});
                prefetch_rows<kT, T, 4>(nl, a.H, nh, t, {static_cast<const T*>(a.k), static_cast<const T*>(a.q), static_cast<const T*>(a.v),
                                                         static_cast<const T*>(a.d_o)});
            }
        }
        if (t == kCopy) ptx::bulk_wait_read0();     // the previous tile's W' has been read out
        bool out_of_form;
        {
            LogSum run = {0.f, 0.f};
            float lo = 0.f, hi = 0.f;
#pragma unroll
            for (int i = 0; i < 16; ++i) run = run + G[i];
            sSeg[seg * 128 + c] = run.hi;
            sSeg[512 + seg * 128 + c] = run.lo;
            __syncthreads();
            LogSum g = {0.f, 0.f}, total = {0.f, 0.f};
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                if (s == seg) g = total;
                total = total + sSeg[s * 128 + c];
                total.lo += sSeg[512 + s * 128 + c];
            }
            const LogSum gm = {0.5f * total.hi, 0.5f * total.lo};
            float* sG = reinterpret_cast<float*>(sm + O_G);
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                const int r = seg * 16 + i;
                g = g + G[i];
                lo = fminf(lo, g.hi); hi = fmaxf(hi, g.hi);
                const float f1 = exp_of(g - gm);
                tile[bt::F + r * kD + c] = f1;
                sG[r * 132 + c] = f1;
            }
            // (a token that is not finite would spoil the earlier ones of its chunk: zeros of a triangle times an infinity)
            uint32_t seen = 0u;
#pragma unroll
            for (int j = 0; j < 2; ++j) { look(seen, kr[j]); look(seen, qr[j]); look(seen, dr[j]); look(seen, vr[j]); }
            const float b = sBeta[t & 63];
            out_of_form = !(lo >= -kBwdRange && hi <= 1.f && total.hi - total.hi == 0.f && b - b == 0.f) || seen_odd<T>(seen);
            if (out_of_form) a.seq_heads[head] = 1;
            if (seg == 0) {
                tile[bt::GC + c] = exp_of(total);
                tile[bt::EM + c] = exp_of(gm);
            }
            if (t < 64) tile[bt::BE + t] = sBeta[t];
        }
        // A head that the sequential kernels do needs no tiles: they are left here (4096 x 32 heads, all of them out of
        // range: the stage 326 us when they went on).
        if (__syncthreads_or(out_of_form || marked)) {
            id += gridDim.x;
            if (!kLoop || id >= n_tiles) break;
            request();
            request_rows();
            request_v();
            continue;
        }
        {
            const float* sG = reinterpret_cast<const float*>(sm + O_G);
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const int r = row0 + 32 * j;
                float kk[8], qq[8], ki[8];
                to_f(kr[j], kk);
                to_f(qr[j], qq);
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const float f1 = sG[r * 132 + c8 + e];
                    ki[e] = kk[e] * reciprocal(f1);
                    kk[e] *= f1;
                    qq[e] *= a.scale * f1;
                }
                put8<128, 2>(sm + O_RQ, r, c8, kk);
                put8<128, 2>(sm + O_RQ, 64 + r, c8, qq);
                put8<64, 2>(sm + O_RK, r, c8, ki);
                if (kExact) put_exact(sm + O_DO, r, c8, dr[j]);
            }
        }
        publish();
        if (w == kIssue) {
            mma6<8>(tm + C_A, k_major<128, 2>(sm + O_RQ), k_major<64, 2>(sm + O_RK), ptx::umma_idesc_bf16(128, 64), false);
            ptx::umma_commit(&bar[0]);
        }
        if (t == kCopy) {
            ptx::bulk_s2g(tile + bt::KI, sm + O_RK, 49152);
            ptx::bulk_commit();
        }
        id += gridDim.x;
        if (kLoop && id < n_tiles) {       // (all but V of this tile has been read from the registers)
            request();
            request_rows();
        }
        float* sL = reinterpret_cast<float*>(sm + O_L);
        float* sT = reinterpret_cast<float*>(sm + O_T);
        for (int idx = t; idx < 64 * LM; idx += kT) sT[idx] = 0.f;
        wait(0);
        // B, L = B Diag(beta) and P: row lane + 32 quad of [B ; P], columns j0 .. j0 + 15
        const int quad = w & 3;
        const uint32_t tq = tm + ((uint32_t)(quad * 32) << 16);
        {
            const int i = (quad & 1) * 32 + lane, j0 = (w >> 2) * 16;
            uint32_t y[16];
            ptx::tmem_ld_32x32b_x16(tq + C_A + j0, y);
            ptx::tmem_ld_wait();
            float v[16];
            const int strict = quad < 2 ? 1 : 0;
#pragma unroll
            for (int e = 0; e < 16; ++e) v[e] = j0 + e + strict <= i ? __uint_as_float(y[e]) : 0.f;
            if (quad < 2) {
#pragma unroll
                for (int e = 0; e < 16; e += 4) {
                    *reinterpret_cast<float4*>(tile + bt::B + i * 64 + j0 + e) = make_float4(v[e], v[e + 1], v[e + 2], v[e + 3]);
                    const float4 b = *reinterpret_cast<const float4*>(sBeta + j0 + e);
                    *reinterpret_cast<float4*>(sL + i * LM + j0 + e) =
                        make_float4(v[e] * b.x, v[e + 1] * b.y, v[e + 2] * b.z, v[e + 3] * b.w);
                }
            } else {
                float x[8];
#pragma unroll
                for (int hf = 0; hf < 2; ++hf) {
#pragma unroll
                    for (int e = 0; e < 8; ++e) x[e] = v[8 * hf + e];
                    put8<64, 1>(sm + O_RP, i, j0 + 8 * hf, x);
                }
            }
        }
        if (t == kCopy) ptx::bulk_wait_read0();
        if (!kExact) {
            __syncthreads();      // K_ has been read out
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                float x[8];
                to_f(dr[j], x);
                put8<64, 2>(sm + O_RK, row0 + 32 * j, c8, x);
            }
        }
        publish();
        if (w == kIssue) {
            const Operand dO = mn_major<64, 2>(sm + (kExact ? O_DO : O_RK));
            mma6<4, kExact>(tm + C_N, dO, mn_major<128, 2>(sm + O_RQ, 64), ptx::umma_idesc_bf16(128, 128) | mnA | mnB, false);
            mma6<4, kExact>(tm + C_X, dO, mn_major<64, 1>(sm + O_RP), ptx::umma_idesc_bf16(128, 64) | mnA | mnB, false);
            ptx::umma_commit(&bar[1]);
        }
        if (w < 4) mma3::invert_unit_lower<LM>(sL, sT, t, [] { ptx::named_bar_sync(1, 128); });
        wait(1);
        __syncthreads();
        {   // T' to the tile and as image; V
            const int r = t >> 3, x0 = (t & 7) * 8;
            float x[8];
#pragma unroll
            for (int e = 0; e < 8; ++e) x[e] = sT[r * LM + x0 + e];
            *reinterpret_cast<float4*>(tile + bt::T + r * 64 + x0) = make_float4(x[0], x[1], x[2], x[3]);
            *reinterpret_cast<float4*>(tile + bt::T + r * 64 + x0 + 4) = make_float4(x[4], x[5], x[6], x[7]);
            put8<64, 1>(sm + O_RP, r, x0, x);
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                if (kExact) {
                    put_exact(sm + O_RK, row0 + 32 * j, c8, vr[j]);
                } else {
                    to_f(vr[j], x);
                    put8<64, 2>(sm + O_RK, row0 + 32 * j, c8, x);
                }
            }
        }
        publish();
        if (w == kIssue) {
            const uint32_t idesc = ptx::umma_idesc_bf16(128, 64) | mnA;
            mma6<4>(tm + C_W, mn_major<128, 2>(sm + O_RQ), k_major<64, 1>(sm + O_RP), idesc, false);
            ptx::umma_commit(&bar[2]);
            mma6<4, kExact>(tm + C_U, mn_major<64, 2>(sm + O_RK), k_major<64, 1>(sm + O_RP), idesc, false);
            ptx::umma_commit(&bar[3]);
        }
        if (kLoop && id < n_tiles) request_v();
        // accumulators out: this thread's row, 16 columns from cg (of N also 64 + cg)
        const int row = quad * 32 + lane, cg = (w >> 2) * 16;
        auto store_rf = [&](uint32_t col, float* m, int c0) {
            uint32_t y[16];
            ptx::tmem_ld_32x32b_x16(tq + col + c0, y);
            ptx::tmem_ld_wait();
#pragma unroll
            for (int e = 0; e < 16; e += 4)
                *reinterpret_cast<uint4*>(m + rf(128, row, c0 + e)) = make_uint4(y[e], y[e + 1], y[e + 2], y[e + 3]);
        };
        store_rf(C_N, tile + bt::N, cg);
        store_rf(C_N, tile + bt::N, 64 + cg);
        store_rf(C_X, tile + bt::X, cg);
        wait(2);              // nothing reads [K^ ; Q] any more: W'^T over it
        {
            uint32_t yw[16];
            ptx::tmem_ld_32x32b_x16(tq + C_W + cg, yw);
            ptx::tmem_ld_wait();
#pragma unroll
            for (int q8 = 0; q8 < 2; ++q8) {
                float x[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) x[e] = __uint_as_float(yw[8 * q8 + e]);
                put8<128, 1>(sm + O_RQ, row, cg + 8 * q8, x);
            }
        }
        publish();
        if (t == kCopy) {
            ptx::bulk_s2g(tile + bt::WI, sm + O_RQ, 49152);
            ptx::bulk_commit();
        }
        wait(3);
        store_rf(C_U, tile + bt::R, cg);
        phase ^= 1u;
        if (!kLoop || id >= n_tiles) break;
    }
    ptx::grid_dep_launch();
    if (w == kIssue && __any_sync(0xffffffffu, !ok)) {      // (not all of the groups issued since have been waited for)
        ptx::umma_commit(done);
        ptx::mbar_wait(done, 0, a.wait_limit_ns);
        __syncwarp();
    }
    if (t == kCopy) ptx::bulk_wait_all0();
    if (!ok && atomicCAS(&a.hdr->status, 0, (int)KDA_ERR_TIMEOUT) == 0) a.hdr->where = 31;
    ptx::tc_fence_before();
    __syncthreads();
    if (w == 0) ptx::tmem_dealloc(tm, 512);
}

}  // namespace

kda_status_t launch_bwd_intra(const BwdChunkArgs& a, kda_dtype_t dt, cudaStream_t st)
{
    {
        DeviceLock lk;
        if (!lk.st) return lk.rc;
        if (!lk.st->attr_done[13]) {
            KDA_CUDA_TRY(cudaFuncSetAttribute(kda_bwd_intra<float>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem));
            KDA_CUDA_TRY(cudaFuncSetAttribute(kda_bwd_intra<__nv_bfloat16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem));
            lk.st->attr_done[13] = true;
        }
    }
    const unsigned tiles = (unsigned)(a.n_chunks * a.H);
    ProfScope ps(PROF_INTRA, st);
    const unsigned loop = tiles < (unsigned)a.n_sm ? tiles : (unsigned)a.n_sm;
    if (dt == KDA_BF16) KDA_CUDA_TRY(launch_dependent(kda_bwd_intra<__nv_bfloat16>, dim3(loop), kT, kSmem, st, a));
    else KDA_CUDA_TRY(launch_dependent(kda_bwd_intra<float>, dim3(tiles), kT, kSmem, st, a));
    count_launch();
    return KDA_OK;
}

}  // namespace kda
