// qs_wide.cu -- launches of the wide fused pass on one state (complex64, 64
// amplitudes per thread; qs_wide_device.cuh holds the pass itself).
#include "qs_wide_device.cuh"

namespace qs {

// FOLD: the circuit's first pass (the uniform state with the folded
// diagonal prefix is generated); the other passes carry none of that code.
template <bool FULL, bool FOLD>
__global__ void __launch_bounds__(kWideThreads, 3)
k_wide_pass(float2 *__restrict__ amps, const WidePass *__restrict__ pass_g, const WideOp *__restrict__ ops_g,
            const uint8_t *__restrict__ codes_g, uint32_t ntiles, FoldArgs fold)
{
    extern __shared__ __align__(16) unsigned char smem_dyn[];
    __shared__ WideSmem S;
    // contiguous range of tiles per CTA
    const uint32_t per = ntiles / gridDim.x, extra = ntiles % gridDim.x;
    const uint32_t t_begin = blockIdx.x * per + (blockIdx.x < extra ? blockIdx.x : extra);
    const uint32_t t_end = t_begin + per + (blockIdx.x < extra ? 1 : 0);
    if constexpr (FOLD) {
        __shared__ WideFoldSmem F;
        if (threadIdx.x == 0) {
#pragma unroll
            for (int i = 0; i < kMaxQubits; ++i) F.nb[i] = fold.nb[i];
            F.m[0] = fold.m1;
            F.m[1] = fold.m2;
            F.m[2] = fold.m4;
        }
        wide_pass_body<FULL, true, false>(amps, pass_g, ops_g, codes_g, t_begin, t_end, S, &F, smem_dyn);
    } else {
        wide_pass_body<FULL, false, false>(amps, pass_g, ops_g, codes_g, t_begin, t_end, S, nullptr, smem_dyn);
    }
}

qs_status run_wide_plan(qs_state *s, const std::vector<WidePass> &passes, size_t nops, const void *dev,
                        double uniform, const FoldArgs *fold)
{
    const FoldArgs none{};
    const WidePass *dpass = static_cast<const WidePass *>(dev);
    const WideOp *dops = reinterpret_cast<const WideOp *>(dpass + passes.size());
    const uint8_t *dcodes = reinterpret_cast<const uint8_t *>(dops + nops);
    for (size_t p = 0; p < passes.size(); ++p) {
        const WidePass &P = passes[p];
        const bool first = p == 0 && uniform != 0.0;
        auto kern = P.full ? (first ? k_wide_pass<true, true> : k_wide_pass<true, false>)
                           : (first ? k_wide_pass<false, true> : k_wide_pass<false, false>);
        const size_t smem = (size_t(1) << P.t) * sizeof(float2);
        QS_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        const uint32_t ntiles = 1u << (P.n - P.t), cap = (uint32_t)s->num_sms * 3;
        kern<<<(int)(ntiles < cap ? ntiles : cap), 1 << (P.t - kWideRegBits), smem, s->stream>>>(
            (float2 *)s->amps, dpass + p, dops, dcodes, ntiles, first && fold ? *fold : none);
        QS_LAUNCH_CHECK();
    }
    return QS_OK;
}

QS_CHECK_READER(check_poll_wide)

}  // namespace qs
