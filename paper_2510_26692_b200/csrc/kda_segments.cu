// Long sequences of few chains (bf16): the chain of a sequence is cut into P segments that run side by side.  A
// segment is an affine map of the state, S_out = A S_in + B, and the chain kernel finds both parts by itself: B as
// the final state from a zero state (from S0 for the first segment), A as the final state from the identity with
// U = 0.  The kernel here then carries the states over the segment borders, S_{p+1} = A_p S_p + B_p, and the chain
// kernel runs once more from them where outputs are wanted.  Twice to three times the chain work, on SMs that had
// none.
//
// One CTA per (8- or 16-column slice, chain), sequential over the segments; products on split tf32 operands
// (kda_mma3.cuh: fp32 accuracy), A fetched one segment ahead.  Bound by the chain of borders (1.5 us each).
//
// Prefill of 8 heads x 4096 tokens 101 -> 72 us, 8 x 30000: 627 -> 256; 16 x 65536 for the final state 1246 -> 656.
#include "kda_common.cuh"
#include "kda_mma3.cuh"
#include "kda_ptx.cuh"

namespace kda {
namespace {

using namespace mma3;
constexpr int kT = 256, LA = 132;
constexpr int kA = 128 * LA;                              // floats of one A
constexpr size_t kSmem = (size_t)(2 * kA + 128 * 24) * 4;

template <int NS>      // columns of a slice
__global__ void __launch_bounds__(kT, 1) kda_segment_states(const __grid_constant__ FusedArgs f, int final_state)
{
    constexpr int LS = NS == 8 ? 8 : NS + 8, NT = NS / 8;
    extern __shared__ __align__(16) float sm[];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5, g = lane >> 2;
    const int col0 = blockIdx.x * NS, job = blockIdx.y;
    float* sS = sm + 2 * kA;
    auto run = [&](int r) { return f.seg_scratch + ((size_t)job * f.seg_runs + r) * (kD * kD); };
    auto fetch = [&](int p) {
        const float* A = run(f.seg_val + p - 1);
        float* d = sm + (p & 1) * kA;
        for (int i = t; i < 128 * 32; i += kT) cp16(d + (i >> 5) * LA + (i & 31) * 4, A + i * 4);
        cp_commit();
    };
    ptx::grid_dep_wait();
    const int last = final_state ? f.seg_P - 1 : f.seg_P - 2;
    if (last >= 1) fetch(1);
    for (int i = t; i < 128 * NS / 4; i += kT) {
        const int r = i / (NS / 4), x = i % (NS / 4) * 4;
        *reinterpret_cast<float4*>(sS + r * LS + x) = *reinterpret_cast<const float4*>(run(0) + r * kD + col0 + x);
    }
    for (int p = 1; p <= last; ++p) {
        float acc[1][NT][4];
        float* b = run(p) + col0;
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
            for (int hf = 0; hf < 2; ++hf) {
                const float2 v = *reinterpret_cast<const float2*>(b + (16 * w + 8 * hf + g) * kD + 8 * nt + 2 * (lane & 3));
                acc[0][nt][2 * hf] = v.x; acc[0][nt][2 * hf + 1] = v.y;
            }
        cp_wait0();
        __syncthreads();
        if (p < last) fetch(p + 1);
        gemm<0, NT, false, false, false, false>(acc, sm + (p & 1) * kA + 16 * w * LA, LA, sS, LS, 0, kD, lane);
        __syncthreads();
        float* out = b;      // the state entering segment p + 1, in the place of B_p
        if (p == last && final_state) {
            const int rank = job / f.a.H, h = job - rank * f.a.H, n = f.ordered ? (int)f.order[rank] : f.n_begin + rank;
            out = f.a.S_out + ((size_t)n * f.a.H + h) * (kD * kD) + col0;
        }
        each_pair(acc, lane, [&](int i, int j, float x, float y) {
            st2(sS + (16 * w + i) * LS + j, x, y);
            st2(out + (16 * w + i) * kD + j, x, y);
        });
    }
}

}  // namespace

kda_status_t launch_segment_states(const FusedArgs& f, int n_count, bool final_state, cudaStream_t st)
{
    {
        DeviceLock lk;
        if (!lk.st) return lk.rc;
        if (!lk.st->attr_done[9]) {
            KDA_CUDA_TRY(cudaFuncSetAttribute(kda_segment_states<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem));
            KDA_CUDA_TRY(cudaFuncSetAttribute(kda_segment_states<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem));
            lk.st->attr_done[9] = true;
        }
    }
    int n_sm = 0;
    if (const kda_status_t rc = sm_count(&n_sm)) return rc;
    const bool narrow = kD / 8 * n_count * f.a.H <= n_sm;     // slices of 8 columns while each has an SM: a shorter step
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(kD / (narrow ? 8 : 16), (unsigned)(n_count * f.a.H));
    cfg.blockDim = dim3(kT);
    cfg.dynamicSmemBytes = kSmem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    ProfScope ps(PROF_INTER, st);
    KDA_CUDA_TRY(cudaLaunchKernelEx(&cfg, narrow ? kda_segment_states<8> : kda_segment_states<16>, f, final_state ? 1 : 0));
    count_launch();
    return KDA_OK;
}

}  // namespace kda
