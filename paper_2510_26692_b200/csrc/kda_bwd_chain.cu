// The two state recurrences of the chunkwise backward pass (equations in kda_bwd_chunk.cu), side by side:
//   forward   r  = U' - W' S            S   <- e^(G_C) S + K~^T (beta r)
//   backward  dX = P^T dO + K~ Lam      Lam <- e^(G_C) Lam + Q^T dO - W'^T (beta dX)       (W', Q here with e^G)
// One CTA per (direction, head, sequence), sequential over the chunks, on tcgen05 with split operands (kda_split3.cuh).
// Everything is transposed: the TMEM lanes are the 128 columns of the state, so that the state and r or dX are A operands
// in TMEM and only what the per-chunk stage left is read from shared memory:
//   D1[v][token] = state^T (W'^T or K_^T)        48 MMAs of N = 64
//   D3[v][k]     = (beta r or -beta dX)^T (K_ or W')       24 of N = 128
// The fp32 state stays in registers (thread = column v, a quarter of k); its operand carries the factor e^(G_m) that W' and K_
// are relative to.  Bound by the chain: 3072 clocks of MMAs a step at least, and the splitting of two operands between
// them.
//
// Warps 0-15 compute (TMEM lane quadrant = warp & 3, quarter of k and of the tokens = warp >> 2), 16 issues the MMAs, 17 loads.
// Each product's operand image has one buffer and the vectors two, requested again when what read them last is known to be
// done.  The state leaves for the tile by way of a buffer of its own.
//
// T=4096, H=32: 570 us with warp-level tf32 products; with state and r in shared memory and two CTAs of 64 columns 277 (6 KB of
// operands for 32 clocks of an MMA of N = 64).  In this form 290 with half the CTAs; six packed sequences of 8 heads, which
// took two waves then, 75 -> 56.  The products with an operand's first splits run while the others are written (296 -> 291 on
// one machine).  A step: 4.05 us (8000 clocks) with 8 CTAs, 4.25 with 32, 4.6 with 64; of 7700 clocks in a build that took times, 2100 for
// the first product, 1300 to r, 1900 for the second, 2400 to the state.  The tensor pipe is active 40 per cent of the time, shared memory
// half busy all the time; a wait that read a flag beside its barrier cost 400 clocks of it.
#include "kda_bwd.cuh"
#include "kda_split3.cuh"

namespace kda {
namespace {

using namespace split3;
constexpr int kT = 640, kCompute = 512;
constexpr int kRegs = 112, kRegsRest = 32;      // of a compute thread and of the others: 512 x 112 + 128 x 32 <= 640 x 96
constexpr uint32_t kImg = 49152, kStateBytes = bt::kState * 4, kVecBytes = bt::kVec * 4;
constexpr uint32_t O_A = 0, O_B = kImg, O_ST = 2 * kImg, O_N = O_ST + kStateBytes, O_VEC = O_N + kStateBytes, O_BAR = O_VEC + 2 * kVecBytes;
constexpr uint32_t kSmem = O_BAR + 192;      // (the images need 1024-byte alignment, and there is no room to align)
static_assert(kSmem <= 232448, "fits the shared memory of one SM");
static_assert(kVecBytes % 16 == 0 && kStateBytes % 16 == 0 && O_BAR % 8 == 0, "bulk copies and barriers are aligned");
// TMEM columns: the operands (three splits each) and the two products
constexpr uint32_t C_S = 0, kSParts = 64, C_X = 192, kXParts = 32, C_1 = 288, C_3 = 352;

template <bool kFwd>
__device__ __forceinline__ void chain_run(const BwdChunkArgs& a, uint8_t* sm, int n, int h)
{
    uint64_t* fullA = reinterpret_cast<uint64_t*>(sm + O_BAR);
    uint64_t* fullB = fullA + 1;
    uint64_t* fullN = fullB + 1;
    uint64_t* fullV = fullN + 1;         // [2]
    uint64_t* m1 = fullV + 2;            // first product of a chunk complete
    uint64_t* m2 = m1 + 1;               // second
    uint64_t* freed = m2 + 1;            // the state has been read out of the staging buffer
    uint64_t* done = freed + 1;          // all MMAs complete
    uint64_t* s_ready = done + 1;        // [3] 16 warps: a split of the state operand written
    uint64_t* x_ready = s_ready + 3;     // [3] 16 warps: of beta r or -beta dX
    uint64_t* staged = x_ready + 3;      // 16 warps: state written to the staging buffer
    uint64_t* n_read = staged + 1;       // 16 warps: N read
    volatile uint32_t* abort_word = reinterpret_cast<volatile uint32_t*>(n_read + 1);
    uint32_t* slot = const_cast<uint32_t*>(abort_word) + 1;
    const int t = threadIdx.x, lane = t & 31, w = ptx::warp_uniform(t >> 5);
    int64_t g0, nc;
    if (a.cu_seqlens) {
        g0 = a.chunk_cu[n]; nc = a.chunk_cu[n + 1] - g0;
    } else {
        g0 = (int64_t)n * a.chunks_per_seq; nc = a.chunks_per_seq;
    }
    auto tile_of = [&](int64_t i) { return a.tiles + ((size_t)(g0 + (kFwd ? i : nc - 1 - i)) * a.H + h) * bt::kFloats; };

    if (w == 0) {
        ptx::tmem_alloc(slot, 512);
        ptx::tmem_relinquish();
    }
    if (t == 32) {
        for (uint64_t* b = fullA; b <= n_read; ++b) ptx::mbar_init(b, b < s_ready ? 1 : kCompute / 32);
        *abort_word = 0;
        ptx::fence_mbar_init();
    }
    ptx::tc_fence_before();
    __syncthreads();
    ptx::tc_fence_after();
    const uint32_t tm = (uint32_t)ptx::warp_uniform((int)*slot);
    // Once any wait of the CTA has run out nobody waits any more.  The lanes of a warp may find that out apart, and must not part
    // on it, or some would wait for the others in the next warp-wide instruction without a bound: warps that go on together
    // ignore the answer, and leave by votes ahead of the state's update.  (Where the votes stand decides more than that they are
    // there.  4096 x 32 heads, this kernel: at every wait 305 us, at none 297, here 294; 7074 x 4, the call: none 620, here 608.  With
    // lanes leaving on their own it was 288 and 607.)  The shared memory is busy: one access to it where one will do.
    auto wait = [&](uint64_t* bar, int64_t phase) {
        if (ptx::mbar_try(bar, (uint32_t)phase & 1u)) return true;
        if (*abort_word == 0 && ptx::mbar_wait(bar, (uint32_t)phase & 1u, a.wait_limit_ns)) return true;
        *abort_word = 1;
        return false;
    };
    auto wait_warp = [&](uint64_t* bar, int64_t phase) {
        wait(bar, phase);
        __syncwarp();
    };

    if (w < kCompute / 32) {
        ptx::reg_inc<kRegs>();
        const int quad = w & 3, part = w >> 2, v = quad * 32 + lane, k0 = part * 32, j0 = part * 16;
        const uint32_t tq = tm + ((uint32_t)(quad * 32) << 16);
        const size_t sbase = (((size_t)n * a.H + h) * kD + k0) * (size_t)kD + v;
        float* stage = reinterpret_cast<float*>(sm + O_ST);
        float2 S[16];
        const float* init = kFwd ? a.S0 : a.dS_T;
#pragma unroll
        for (int e = 0; e < 16; ++e)
            S[e] = init ? make_float2(init[sbase + (size_t)(2 * e) * kD], init[sbase + (size_t)(2 * e + 1) * kD]) : make_float2(0.f, 0.f);
        // a vector of a chunk's step: four values from c on
        auto vec = [&](int64_t i, int off, int c) {
            return *reinterpret_cast<const float4*>(sm + O_VEC + (uint32_t)(i & 1) * kVecBytes + (uint32_t)(off - bt::GC + c) * 4);
        };
        auto lo = [](const float4& m) { return make_float2(m.x, m.y); };
        auto hi = [](const float4& m) { return make_float2(m.z, m.w); };
        auto pair = [](const uint32_t* y) { return make_float2(__uint_as_float(y[0]), __uint_as_float(y[1])); };
        auto arrive = [&](uint64_t* bar) {
            ptx::tmem_st_wait();
            ptx::tc_fence_before();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(bar);
        };
        auto put_state = [&](int64_t i) {
            wait(&fullV[i & 1], i >> 1);
            float2 x[16];
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const float4 m = vec(i, bt::EM, k0 + 4 * e);
                x[2 * e] = __fmul2_rn(lo(m), S[2 * e]);
                x[2 * e + 1] = __fmul2_rn(hi(m), S[2 * e + 1]);
            }
            put_tmem<kSParts>(tq + C_S + part * 16, x, [&](int s) { arrive(&s_ready[s]); });
        };
        if (nc > 0) put_state(0);
        for (int64_t i = 0; i < nc; ++i) {
            float* tile = tile_of(i);
            float* ux = tile + (kFwd ? bt::R : bt::X) + rf(128, v, j0);
            uint32_t u[16];
#pragma unroll
            for (int e = 0; e < 16; e += 4) ldraw4_w(u + e, ux + e * 128);
            // the state as the gradients stage needs it, by way of shared memory
            if (i > 0) wait(freed, i - 1);
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                stage[sf(k0 + 2 * e, v)] = S[e].x;
                stage[sf(k0 + 2 * e + 1, v)] = S[e].y;
            }
            ptx::fence_async_smem();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(staged);
            wait_warp(m1, i);
            ptx::tc_fence_after();
            {
                uint32_t y[16];
                ptx::tmem_ld_32x32b_x16(tq + C_1 + j0, y);
                ptx::tmem_ld_wait();
                const float sg = kFwd ? -1.f : 1.f;
                float2 x[8], z[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) x[e] = __ffma2_rn(pair(y + 2 * e), make_float2(sg, sg), pair(u + 2 * e));
#pragma unroll
                for (int e = 0; e < 8; e += 2) {
                    float4 b = vec(i, bt::BE, j0 + 2 * e);
                    if (!kFwd) b = make_float4(-b.x, -b.y, -b.z, -b.w);
                    z[e] = __fmul2_rn(lo(b), x[e]);
                    z[e + 1] = __fmul2_rn(hi(b), x[e + 1]);
                }
                put_tmem<kXParts>(tq + C_X + part * 8, z, [&](int s) { arrive(&x_ready[s]); });
#pragma unroll
                for (int e = 0; e < 16; e += 4)
                    *reinterpret_cast<float4*>(ux + e * 128) = make_float4(x[e / 2].x, x[e / 2].y, x[e / 2 + 1].x, x[e / 2 + 1].y);
            }
            // what does not need the second product
            if (!kFwd && !__all_sync(0xffffffffu, wait(fullN, i))) break;
            const float* np = reinterpret_cast<const float*>(sm + O_N) + rf(128, v, k0);
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const float4 gc = vec(i, bt::GC, k0 + 4 * e);
                S[2 * e] = __fmul2_rn(lo(gc), S[2 * e]);
                S[2 * e + 1] = __fmul2_rn(hi(gc), S[2 * e + 1]);
                if (!kFwd) {
                    const float4 em = vec(i, bt::EM, k0 + 4 * e), nn = *reinterpret_cast<const float4*>(np + e * 512);
                    S[2 * e] = __ffma2_rn(lo(em), lo(nn), S[2 * e]);
                    S[2 * e + 1] = __ffma2_rn(hi(em), hi(nn), S[2 * e + 1]);
                }
            }
            if (!kFwd) {
                __syncwarp();
                if (lane == 0) ptx::mbar_arrive(n_read);
            }
            if (!__all_sync(0xffffffffu, wait(m2, i))) break;
            ptx::tc_fence_after();
            {
                uint32_t y[32];
                ptx::tmem_ld_32x32b_x32(tq + C_3 + k0, y);
                ptx::tmem_ld_wait();
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const float4 em = vec(i, bt::EM, k0 + 4 * e);
                    S[2 * e] = __ffma2_rn(lo(em), pair(y + 4 * e), S[2 * e]);
                    S[2 * e + 1] = __ffma2_rn(hi(em), pair(y + 4 * e + 2), S[2 * e + 1]);
                }
            }
            if (i + 1 < nc) put_state(i + 1);
        }
        ptx::tc_fence_before();
        if (!kFwd && a.dS0)
#pragma unroll
            for (int e = 0; e < 16; ++e) {
                a.dS0[sbase + (size_t)(2 * e) * kD] = S[e].x;
                a.dS0[sbase + (size_t)(2 * e + 1) * kD] = S[e].y;
            }
    } else {
        ptx::reg_dec<kRegsRest>();
        if (w == kCompute / 32 + 1) {
            if (lane == 0) {
                auto get = [&](uint32_t at, int64_t j, int from, uint32_t bytes, uint64_t* bar) {
                    ptx::mbar_expect_tx(bar, bytes);
                    ptx::bulk_g2s(sm + at, tile_of(j) + from, bytes, bar);
                };
                auto first = [&](int64_t j) { get(O_A, j, kFwd ? bt::WI : bt::KI, kImg, fullA); };
                auto second = [&](int64_t j) { get(O_B, j, kFwd ? bt::KI : bt::WI, kImg, fullB); };
                auto vectors = [&](int64_t j) { get(O_VEC + (uint32_t)(j & 1) * kVecBytes, j, bt::GC, kVecBytes, &fullV[j & 1]); };
                auto n_of = [&](int64_t j) { if (!kFwd) get(O_N, j, bt::N, kStateBytes, fullN); };
                // what the compute warps read themselves, asked into L2 two steps ahead
                auto ahead = [&](int64_t j) { if (j < nc) prefetch_l2(tile_of(j) + (kFwd ? bt::R : bt::X), 64 * kD * 4); };
                int64_t in_a = 0, in_b = 0, in_n = 0;      // requested so far (vectors with the first operand)
                if (nc > 0) {
                    vectors(0); first(0); second(0); n_of(0);
                    in_a = in_b = in_n = 1;
                }
                ahead(1);
                for (int64_t i = 0; i < nc; ++i) {
                    const bool more = i + 1 < nc;
                    if (!wait(staged, i)) break;
                    ptx::bulk_s2g(tile_of(i) + (kFwd ? bt::S : bt::L), sm + O_ST, kStateBytes);
                    ptx::bulk_commit();
                    if (!wait(m1, i)) break;
                    if (more) {        // (the first product's operand is free, and so are the vectors of chunk i - 1)
                        vectors(i + 1); first(i + 1);
                        ++in_a;
                    }
                    ahead(i + 2);
                    ptx::bulk_wait_read0();
                    ptx::mbar_arrive(freed);
                    if (!kFwd) {
                        if (!wait(n_read, i)) break;
                        if (more) { n_of(i + 1); ++in_n; }
                    }
                    if (!wait(m2, i)) break;
                    if (more) { second(i + 1); ++in_b; }
                }
                ptx::bulk_wait_all0();
                if (*abort_word) {      // nothing may be in flight when the CTA leaves
                    for (int64_t j = in_a > 1 ? in_a - 2 : 0; j < in_a; ++j) ptx::mbar_wait(&fullV[j & 1], (uint32_t)(j >> 1) & 1u, a.wait_limit_ns);
                    if (in_a > 0) ptx::mbar_wait(fullA, (uint32_t)(in_a - 1) & 1u, a.wait_limit_ns);
                    if (in_b > 0) ptx::mbar_wait(fullB, (uint32_t)(in_b - 1) & 1u, a.wait_limit_ns);
                    if (!kFwd && in_n > 0) ptx::mbar_wait(fullN, (uint32_t)(in_n - 1) & 1u, a.wait_limit_ns);
                }
            }
        } else if (w == kCompute / 32) {
            const uint32_t id64 = ptx::umma_idesc_bf16(128, 64), id128 = ptx::umma_idesc_bf16(128, 128), mnB = ptx::kIdescBMajorMN;
            for (int64_t i = 0; i < nc; ++i) {
                // the products with the first splits of an operand run while the others are written
                auto operand = [&](uint64_t* ready) {
                    return [&, ready](int s) {
                        wait_warp(&ready[s], i);
                        ptx::tc_fence_after();
                    };
                };
                wait(fullA, i);
                mma6_ta<8, kSParts>(tm + C_1, tm + C_S, kFwd ? mn_major<128, 1>(sm + O_A) : k_major<64, 2>(sm + O_A), kFwd ? id64 | mnB : id64, false, operand(s_ready));
                ptx::umma_commit(m1);
                wait(fullB, i);
                mma6_ta<4, kXParts>(tm + C_3, tm + C_X, kFwd ? mn_major<64, 2>(sm + O_B) : k_major<128, 1>(sm + O_B), kFwd ? id128 | mnB : id128, false, operand(x_ready));
                ptx::umma_commit(m2);
            }
            __syncwarp();
            ptx::umma_commit(done);        // before the TMEM goes away
            if (!ptx::mbar_wait(done, 0, a.wait_limit_ns)) *abort_word = 1;
            __syncwarp();
        }
    }
    ptx::grid_dep_launch();
    __syncthreads();
    if (t == 0 && *abort_word && atomicCAS(&a.hdr->status, 0, (int)KDA_ERR_TIMEOUT) == 0) a.hdr->where = 32;
    if (w == 0) ptx::tmem_dealloc(tm, 512);
}

__global__ void __launch_bounds__(kT, 1) kda_bwd_chain(BwdChunkArgs a)
{
    extern __shared__ __align__(1024) uint8_t sm[];
    const int h = blockIdx.y, n = blockIdx.z;
    ptx::grid_dep_wait();      // (launched before the preceding kernel has ended)
    if (a.seq_heads[h]) return;
    if ((ptx::smem_u32(sm) & 1023u) != 0) {
        if (threadIdx.x == 0 && atomicCAS(&a.hdr->status, 0, (int)KDA_ERR_CUDA) == 0) a.hdr->where = 33;
        return;
    }
    if (blockIdx.x & 1) chain_run<true>(a, sm, n, h);
    else chain_run<false>(a, sm, n, h);
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
    KDA_CUDA_TRY(launch_dependent(kda_bwd_chain, dim3(2, (unsigned)a.H, (unsigned)a.n_seqs), kT, kSmem, st, a));
    count_launch();
    return KDA_OK;
}

}  // namespace kda
