// The two state recurrences of the chunkwise backward pass (equations in kda_bwd_chunk.cu), side by side:
//   forward   r  = U' - W' S            S   <- e^(G_C) S + K~^T (beta r)
//   backward  dX = P^T dO + K~ Lam      Lam <- e^(G_C) Lam + Q^T dO - W'^T (beta dX)       (W', Q here with e^G)
// State columns never mix: one CTA per (64-column slice, direction, head, sequence), sequential over the chunks,
// on tcgen05 with split operands (kda_split3.cuh).  The fp32 state stays in registers (thread = row, half of
// the columns); its operand image carries the factor e^(G_m) that W' and K_ are relative to.  Bound by the
// chain: two dependent groups of MMAs (48 and 24 of N = 64) with their read-outs per chunk.
//
// Warps 0-7 compute (TMEM lane quadrant = warp & 3, column half = warp >> 2), 8 issues the MMAs, 9 loads.
// The first product's operand image has two buffers, the second's one: each is requested when the product
// that read it last is complete, most of a step ahead.
//
// T=4096, H=32 (128 CTAs): 570 us with warp-level tf32 products, 323 in this form.
#include "kda_bwd.cuh"
#include "kda_split3.cuh"

namespace kda {
namespace {

using namespace split3;
constexpr int kT = 320;
constexpr int NS = 64;
constexpr uint32_t kImg = 49152;
constexpr uint32_t O_A = 0, O_B = 2 * kImg, O_S = 3 * kImg, O_X = 4 * kImg, O_BAR = O_X + 24576;
constexpr uint32_t kSmem = O_BAR + 128 + 1024;
static_assert(kSmem <= 232448, "fits the shared memory of one SM");
constexpr uint32_t C_1 = 0, C_2 = NS;      // TMEM columns of the two products

template <bool kFwd>
__device__ __forceinline__ void chain_run(const BwdChunkArgs& a, uint8_t* sm, int n, int h, int col0)
{
    uint64_t* fullA = reinterpret_cast<uint64_t*>(sm + O_BAR);   // [2]
    uint64_t* fullB = fullA + 2;
    uint64_t* m1 = fullB + 1;            // first product of a chunk complete
    uint64_t* m2 = m1 + 1;               // second
    uint64_t* s_ready = m2 + 1;          // 8 warps: state image written
    uint64_t* x_ready = s_ready + 1;     // 4 warps: beta r or -beta dX written
    volatile uint32_t* abort_word = reinterpret_cast<volatile uint32_t*>(x_ready + 1);
    uint32_t* slot = const_cast<uint32_t*>(abort_word) + 1;
    const int t = threadIdx.x, lane = t & 31, w = ptx::warp_uniform(t >> 5);
    int64_t g0, nc, tok_begin, tok_end;
    if (a.cu_seqlens) {
        g0 = a.chunk_cu[n]; nc = a.chunk_cu[n + 1] - g0;
        tok_begin = a.cu_seqlens[n]; tok_end = a.cu_seqlens[n + 1];
    } else {
        g0 = (int64_t)n * a.chunks_per_seq; nc = a.chunks_per_seq;
        tok_begin = (int64_t)n * a.seq_len; tok_end = tok_begin + a.seq_len;
    }
    auto chunk_of = [&](int64_t i) { return kFwd ? i : nc - 1 - i; };
    auto tile_of = [&](int64_t i) { return a.tiles + ((size_t)(g0 + chunk_of(i)) * a.H + h) * bt::kFloats; };

    if (w == 0) {
        ptx::tmem_alloc(slot, 128);
        ptx::tmem_relinquish();
    }
    if (t == 32) {
        ptx::mbar_init(&fullA[0], 1);
        ptx::mbar_init(&fullA[1], 1);
        ptx::mbar_init(fullB, 1);
        ptx::mbar_init(m1, 1);
        ptx::mbar_init(m2, 1);
        ptx::mbar_init(s_ready, 8);
        ptx::mbar_init(x_ready, 4);
        *abort_word = 0;
        ptx::fence_mbar_init();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tm = (uint32_t)ptx::warp_uniform((int)*slot);
    // false once any wait of the CTA has run out
    auto wait = [&](uint64_t* bar, int64_t phase) {
        if (!ptx::mbar_wait(bar, (uint32_t)phase & 1u, a.wait_limit_ns)) *abort_word = 1;
        return *abort_word == 0;
    };

    if (w == 9) {
        if (lane == 0) {
            int64_t i = 0;
            // what a step reads into registers, asked into L2 two steps ahead: 64 rows of R or X, 128 of N, the vectors
            auto ahead = [&](int64_t j) {
                if (j >= nc) return;
                const float* p = tile_of(j);
                prefetch_l2(p + (kFwd ? bt::R : bt::X) + rf(64, 0, col0), 64 * NS * 4);
                if (!kFwd) prefetch_l2(p + bt::N + rf(128, 0, col0), 128 * NS * 4);
                prefetch_l2(p + bt::GC, 256 * 4);
            };
            ahead(1);
            for (; i < nc; ++i) {
                const float* tile = tile_of(i);
                ahead(i + 2);
                // (i >= 2: the second product of chunk i - 2 has been waited for below, and with it the first, which
                // read this buffer.  The barrier of the first may be a phase further on by now.)
                ptx::mbar_expect_tx(&fullA[i & 1], kImg);
                ptx::bulk_g2s(sm + O_A + (i & 1) * kImg, tile + (kFwd ? bt::WI : bt::KI), kImg, &fullA[i & 1]);
                if (i >= 1 && !wait(m2, i - 1)) { ++i; break; }
                ptx::mbar_expect_tx(fullB, kImg);
                ptx::bulk_g2s(sm + O_B, tile + (kFwd ? bt::KI : bt::WI), kImg, fullB);
            }
            if (*abort_word) {      // nothing may be in flight when the CTA leaves
                for (int64_t j = i > 2 ? i - 2 : 0; j < i; ++j) ptx::mbar_wait(&fullA[j & 1], (uint32_t)(j >> 1) & 1u, a.wait_limit_ns);
                for (int64_t j = i > 2 ? i - 2 : 0; j < i; ++j) ptx::mbar_wait(fullB, (uint32_t)j & 1u, a.wait_limit_ns);
            }
        }
    } else if (w == 8) {
        const uint32_t id1 = ptx::umma_idesc_bf16(128, NS) | ptx::kIdescBMajorMN, id2 = id1 | ptx::kIdescAMajorMN;
        for (int64_t i = 0; i < nc; ++i) {
            if (!wait(s_ready, i) || !wait(&fullA[i & 1], i >> 1)) break;
            __syncwarp();
            ptx::tc_fence_after();
            mma6<8>(tm + C_1, k_major<64, 2>(sm + O_A + (i & 1) * kImg), mn_major<128, 1>(sm + O_S), id1, false);
            ptx::umma_commit(m1);
            if (!wait(x_ready, i) || !wait(fullB, i)) break;
            __syncwarp();
            ptx::tc_fence_after();
            mma6<4>(tm + C_2, mn_major<64, 2>(sm + O_B), mn_major<64, 1>(sm + O_X), id2, false);
            ptx::umma_commit(m2);
        }
    } else {
        const int quad = w & 3, row = quad * 32 + lane, ch = (w >> 2) * 32;
        const uint32_t tq = tm + ((uint32_t)(quad * 32) << 16);
        const size_t sbase = (((size_t)n * a.H + h) * kD + row) * (size_t)kD + col0 + ch;
        const bool rows_x = quad < 2;           // rows 0-63 of the first product are tokens, the rest is not used
        float S[32];
        const float* init = kFwd ? a.S0 : a.dS_T;
#pragma unroll
        for (int e = 0; e < 32; e += 4) {
            const float4 v = init ? *reinterpret_cast<const float4*>(init + sbase + e) : make_float4(0.f, 0.f, 0.f, 0.f);
            S[e] = v.x; S[e + 1] = v.y; S[e + 2] = v.z; S[e + 3] = v.w;
        }
        auto put_state = [&](float em) {
#pragma unroll
            for (int q8 = 0; q8 < 4; ++q8) {
                float x[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) x[e] = em * S[8 * q8 + e];
                put8<128, 1>(sm + O_S, row, ch + 8 * q8, x);
            }
            ptx::fence_async_smem();
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(s_ready);
        };
        float em = nc > 0 ? tile_of(0)[bt::EM + row] : 0.f;
        if (nc > 0) put_state(em);
        for (int64_t i = 0; i < nc; ++i) {
            float* tile = tile_of(i);
            const float em_next = i + 1 < nc ? tile_of(i + 1)[bt::EM + row] : 0.f;
            const float gam = tile[bt::GC + row];
            uint32_t u[32], nn[kFwd ? 1 : 32];
            float beta = 0.f;
            float* ux = tile + (kFwd ? bt::R : bt::X);
            if (rows_x) {
#pragma unroll
                for (int e = 0; e < 32; e += 4) ldraw4_w(u + e, ux + rf(64, row, col0 + ch + e));
                const int64_t tok = tok_begin + chunk_of(i) * kC + row;
                if (tok < tok_end) beta = a.beta[(size_t)tok * a.H + h];
            }
            if (!kFwd)
#pragma unroll
                for (int e = 0; e < (kFwd ? 0 : 32); e += 4) ldraw4(nn + e, tile + bt::N + rf(128, row, col0 + ch + e));
            {   // the state as the gradients stage needs it
                float* keep = tile + (kFwd ? bt::S : bt::L);
#pragma unroll
                for (int e = 0; e < 32; e += 4)
                    *reinterpret_cast<float4*>(keep + rf(128, row, col0 + ch + e)) = make_float4(S[e], S[e + 1], S[e + 2], S[e + 3]);
            }
            if (!wait(m1, i)) break;
            __syncwarp();
            ptx::tc_fence_after();
            if (rows_x) {
                uint32_t y[32];
                ptx::tmem_ld_32x32b_x32(tq + C_1 + ch, y);
                ptx::tmem_ld_wait();
                float x[32];
#pragma unroll
                for (int e = 0; e < 32; ++e)
                    x[e] = kFwd ? __uint_as_float(u[e]) - __uint_as_float(y[e]) : __uint_as_float(u[e]) + __uint_as_float(y[e]);
                const float f = kFwd ? beta : -beta;
#pragma unroll
                for (int q8 = 0; q8 < 4; ++q8) {
                    float z[8];
#pragma unroll
                    for (int e = 0; e < 8; ++e) z[e] = f * x[8 * q8 + e];
                    put8<64, 1>(sm + O_X, row, ch + 8 * q8, z);
                }
                ptx::fence_async_smem();
                ptx::tc_fence_before();
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(x_ready);
#pragma unroll
                for (int e = 0; e < 32; e += 4)
                    *reinterpret_cast<float4*>(ux + rf(64, row, col0 + ch + e)) = make_float4(x[e], x[e + 1], x[e + 2], x[e + 3]);
            }
#pragma unroll
            for (int e = 0; e < 32; ++e) S[e] = kFwd ? S[e] * gam : fmaf(em, __uint_as_float(nn[kFwd ? 0 : e]), S[e] * gam);
            if (!wait(m2, i)) break;
            __syncwarp();
            ptx::tc_fence_after();
            uint32_t y[32];
            ptx::tmem_ld_32x32b_x32(tq + C_2 + ch, y);
            ptx::tmem_ld_wait();
#pragma unroll
            for (int e = 0; e < 32; ++e) S[e] = fmaf(em, __uint_as_float(y[e]), S[e]);
            em = em_next;
            if (i + 1 < nc) put_state(em);
        }
        ptx::tc_fence_before();
        if (!kFwd && a.dS0)
#pragma unroll
            for (int e = 0; e < 32; e += 4)
                *reinterpret_cast<float4*>(a.dS0 + sbase + e) = make_float4(S[e], S[e + 1], S[e + 2], S[e + 3]);
    }
    __syncthreads();
    if (t == 0 && *abort_word && atomicCAS(&a.hdr->status, 0, (int)KDA_ERR_TIMEOUT) == 0) a.hdr->where = 32;
    if (w == 0) ptx::tmem_dealloc(tm, 128);
}

__global__ void __launch_bounds__(kT, 1) kda_bwd_chain(BwdChunkArgs a)
{
    extern __shared__ uint8_t smem_raw[];
    const int h = blockIdx.y, n = blockIdx.z, slice = blockIdx.x >> 1;
    if (a.seq_heads[h]) return;
    uint8_t* sm = smem_raw + ((1024u - (ptx::smem_u32(smem_raw) & 1023u)) & 1023u);
    if (blockIdx.x & 1) chain_run<true>(a, sm, n, h, slice * NS);
    else chain_run<false>(a, sm, n, h, slice * NS);
}

}  // namespace

kda_status_t launch_bwd_chain(const BwdChunkArgs& a, cudaStream_t st)
{
    {
        DeviceLock lk;
        if (!lk.st) return lk.rc;
        if (!lk.st->attr_done[15]) {
            KDA_CUDA_TRY(cudaFuncSetAttribute(kda_bwd_chain, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem));
            lk.st->attr_done[15] = true;
        }
    }
    ProfScope ps(PROF_INTER, st);
    kda_bwd_chain<<<dim3(2 * kD / NS, (unsigned)a.H, (unsigned)a.n_seqs), kT, kSmem, st>>>(a);
    count_launch();
    KDA_CUDA_TRY(cudaGetLastError());
    return KDA_OK;
}

}  // namespace kda
