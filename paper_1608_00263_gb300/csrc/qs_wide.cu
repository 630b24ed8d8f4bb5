// qs_wide.cu -- launches of the wide fused pass (complex64, 64 amplitudes per
// thread; qs_wide_device.cuh holds the pass itself) on one state and in the
// batch engines.
#include "qs_stats_device.cuh"
#include "qs_wide_device.cuh"

namespace qs {

// FOLD: the circuit's first pass (the uniform state with the folded
// diagonal prefix is generated); the other passes carry none of that code.
template <bool FULL, bool FOLD, int RB>
__global__ void __launch_bounds__(1 << (13 - RB), RB == kWideRegBits ? 3 : 2)
k_wide_pass(float2 *__restrict__ amps, const WidePass *__restrict__ pass_g, const WideOp *__restrict__ ops_g,
            const uint8_t *__restrict__ codes_g, uint32_t ntiles, FoldArgs fold)
{
    extern __shared__ __align__(16) unsigned char smem_dyn[];
    __shared__ WideSmemT<RB> S;
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
            F.plain = fold.nfold == 0;
        }
        wide_pass_body<FULL ? 1 : 0, 1, 0, RB>(amps, pass_g, ops_g, codes_g, t_begin, t_end, S, &F, smem_dyn);
    } else {
        wide_pass_body<FULL ? 1 : 0, 0, 0, RB>(amps, pass_g, ops_g, codes_g, t_begin, t_end, S, nullptr, smem_dyn);
    }
}

template <int RB>
static auto wide_pass_kernel(bool full, bool first)
{
    return full ? (first ? k_wide_pass<true, true, RB> : k_wide_pass<true, false, RB>)
                : (first ? k_wide_pass<false, true, RB> : k_wide_pass<false, false, RB>);
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
        auto kern = P.r == kWideRegBits ? wide_pass_kernel<kWideRegBits>(P.full != 0, first)
                                        : wide_pass_kernel<kWideFewRegBits>(P.full != 0, first);
        const size_t smem = (size_t(1) << P.t) * sizeof(float2);
        QS_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kTileBytes));
        const uint32_t ntiles = 1u << (P.n - P.t), cap = (uint32_t)s->num_sms * (P.r == kWideRegBits ? 3 : 2);
        kern<<<(int)(ntiles < cap ? ntiles : cap), 1 << (P.t - P.r), smem, s->stream>>>(
            (float2 *)s->amps, dpass + p, dops, dcodes, ntiles, first && fold ? *fold : none);
        QS_LAUNCH_CHECK();
    }
    return QS_OK;
}

// ---- adjoint sweep: one pass over psi and lambda ----
// Partials: warp w of CTA b adds its sums of slot s at part[s * stride + b *
// (warps per CTA) + w]; each address has one warp, so the order is fixed.
__global__ void __launch_bounds__(kWideThreads, 3)
k_adj_wide(float2 *__restrict__ psi, uint64_t lam_off, const WidePass *__restrict__ pass_g,
           const WideOp *__restrict__ ops_g, const uint8_t *__restrict__ codes_g, uint32_t ntiles, double *part,
           uint32_t stride)
{
    extern __shared__ __align__(16) unsigned char smem_dyn[];
    __shared__ WideSmem S;
    if (threadIdx.x == 0) {
        S.part = reinterpret_cast<uint64_t>(part + (size_t)blockIdx.x * (blockDim.x >> 5));
        S.part_stride = (uint64_t)stride * 8u;
    }
    const uint32_t per = ntiles / gridDim.x, extra = ntiles % gridDim.x;
    const uint32_t t_begin = blockIdx.x * per + (blockIdx.x < extra ? blockIdx.x : extra);
    wide_pass_body<2, 0, 0>(psi, pass_g, ops_g, codes_g, t_begin,
                                    t_begin + per + (blockIdx.x < extra ? 1 : 0), S, nullptr, smem_dyn, lam_off);
}

int adjoint_wide_partials(const qs_state *s) { return 3 * s->num_sms * (kWideThreads / 32); }

qs_status launch_adjoint_wide(const qs_state *s, void *lam, const WidePlan &plan, const void *dev, double *part)
{
    const WidePass *dpass = static_cast<const WidePass *>(dev);
    const WideOp *dops = reinterpret_cast<const WideOp *>(dpass + plan.passes.size());
    const uint8_t *dcodes = reinterpret_cast<const uint8_t *>(dops + plan.ops.size());
    const uint64_t lam_off = (uint64_t)((const char *)lam - (const char *)s->amps);
    for (size_t p = 0; p < plan.passes.size(); ++p) {
        const WidePass &P = plan.passes[p];
        const size_t smem = (size_t(1) << P.t) * sizeof(float2);
        if (p == 0) QS_CUDA_TRY(cudaFuncSetAttribute(k_adj_wide, cudaFuncAttributeMaxDynamicSharedMemorySize, kTileBytes));
        const uint32_t ntiles = 1u << (P.n - P.t), cap = (uint32_t)s->num_sms * 3;
        k_adj_wide<<<(int)(ntiles < cap ? ntiles : cap), 1 << (P.t - kWideRegBits), smem, s->stream>>>(
            (float2 *)s->amps, lam_off, dpass + p, dops, dcodes, ntiles, part, (uint32_t)adjoint_wide_partials(s));
        QS_LAUNCH_CHECK();
    }
    return QS_OK;
}

// ---- batch engines on wide passes ----
// Lockstep round: blockDim.x = 2^(t - 6), the launch's tile size.
template <bool FULL>
__global__ void __launch_bounds__(kWideThreads, 3)
k_batch_pass_wide(float2 *__restrict__ amps, const BatchItem *__restrict__ items, int nitems,
                  const WidePass *__restrict__ passes, const WideOp *__restrict__ ops,
                  const uint8_t *__restrict__ codes, const FoldArgs *__restrict__ folds)
{
    extern __shared__ __align__(16) unsigned char smem_dyn[];
    __shared__ WideSmem S;
    __shared__ WideFoldSmem F;
    for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
        const BatchItem w = items[it];
        wide_pass_body<FULL ? 1 : 0, 2, 0>(amps + w.amp_off, passes + w.pass, ops, codes, w.tile_begin, w.tile_end, S,
                                               &F, smem_dyn, 0, folds);
    }
}

// Sum of an accumulator's partials in slot order, sixteen loads in flight: one
// load after the other cost 0.58 us a slot, 0.6 ms for the 1024 slots of a
// 26-qubit instance, at the end of the run.
__device__ __forceinline__ double sum_slots(const double *part, uint32_t nslots)
{
    double acc = 0;
    for (uint32_t j0 = 0; j0 < nslots; j0 += 16) {
        double v[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = j0 + j < nslots ? __ldcg(part + (size_t)(j0 + j) * kStatAcc) : 0.0;
#pragma unroll
        for (int j = 0; j < 16; ++j)
            if (j0 + j < nslots) acc += v[j];
    }
    return acc;
}

// Persistent engine (PersistItem, see k_batch_persistent): the same queue,
// dependency waits and completion counts with CTAs of kWideThreads threads,
// three per SM.  FULL: some item's pass holds parameterised gates; the loop
// that knows them then runs every pass.  GROUPED as in wide_pass_body.
template <bool FULL, int GROUPED>
__global__ void __launch_bounds__(kWideThreads, 3)
k_batch_persistent_wide(float2 *amps, const PersistItem *__restrict__ items, int nitems,
                        const WidePass *__restrict__ passes, const WideOp *__restrict__ ops,
                        const uint8_t *__restrict__ codes, const FoldArgs *__restrict__ folds, uint32_t *done,
                        PersistCtl *ctl, double *part, double *sums, uint64_t wait_ns)
{
    extern __shared__ __align__(16) unsigned char smem_dyn[];
    __shared__ WideSmem S;
    __shared__ WideFoldSmem F;
    __shared__ int s_item, s_go, s_last;
    __shared__ PersistItem w;        // the item: no registers held across a pass
    for (;;) {
        if (threadIdx.x == 0) {
            s_item = (int)atomicAdd(&ctl->next, 1u);
            if (s_item < nitems) w = items[s_item];
        }
        __syncthreads();
        if (s_item >= nitems) break;
        if (threadIdx.x == 0) {
            int go = *(volatile const uint32_t *)&ctl->abort == 0;
            if (go && w.need) {
                const int r = flag_wait_bounded(done + w.inst, w.need, &ctl->abort, wait_ns);
                if (r == 1) {
                    atomicExch(&ctl->err, 1u);
                    atomicExch(&ctl->abort, 1u);
                }
                go = r == 0;
            }
            s_go = go;
        }
        __syncthreads();
        if (s_go) {
            if (w.kind == kPersistInit) {
                // (lo = 0: the instance's first pass generates its state)
                float4 *a = reinterpret_cast<float4 *>(amps + w.amp_off);
                const float4 u = make_float4(w.f0, 0.f, w.f0, 0.f);
                for (uint32_t e = threadIdx.x; e < w.lo / 2; e += blockDim.x) a[e] = u;
                if (threadIdx.x == 0 && w.lo) a[0] = make_float4(w.f1, 0.f, w.f0, 0.f);
            } else if (w.kind == kPersistStats) {
                batch_stats_chunk<kWideThreads, true>(amps + w.amp_off, w.lo, w.f0, part + (size_t)w.pass * kStatAcc);
            } else {
                wide_pass_body<FULL ? 1 : 0, 2, GROUPED>(amps + w.amp_off, passes + w.pass, ops, codes, w.lo, w.hi, S, &F,
                                                      smem_dyn, 0, folds);
            }
        }
        // Thread 0 overwrites the item once it has taken the next one: the
        // others have read what they need of it before the last barrier.
        const bool stats = w.kind == kPersistStats;
        __syncthreads();
        if (threadIdx.x == 0) {
            __threadfence();
            const uint32_t prev = atomicAdd(done + w.inst, 1u);
            if (stats) {
                s_last = prev + 1 == w.total;
                __threadfence();
            }
        }
        if (stats) {
            __syncthreads();
            if (s_last && threadIdx.x < kStatAcc) {
                sums[(size_t)w.inst * kStatAcc + threadIdx.x] =
                    sum_slots(part + (size_t)w.hi * kStatAcc + threadIdx.x, w.nslots);
            }
            __syncthreads();
        }
    }
}

qs_status launch_batch_round_wide(cudaStream_t st, int num_sms, void *amps, const void *items, int nitems,
                                  int tile_bits, const WidePass *passes, const WideOp *ops, const uint8_t *codes,
                                  const FoldArgs *folds, bool full)
{
    if (tile_bits < kWideMinTile || tile_bits > 13) return set_error(QS_ERR_INVALID_ARG, "batch tile bits %d", tile_bits);
    auto kern = full ? k_batch_pass_wide<true> : k_batch_pass_wide<false>;
    const int cap = num_sms * 3;
    kern<<<nitems < cap ? nitems : cap, 1 << (tile_bits - kWideRegBits), (size_t(1) << tile_bits) * sizeof(float2), st>>>(
        (float2 *)amps, (const BatchItem *)items, nitems, passes, ops, codes, folds);
    QS_LAUNCH_CHECK();
    return QS_OK;
}

// The persistent kernel by (parameterised gates, tiles in groups): with thread
// groups the tile stride, the barrier id and the buffer address are per-thread
// values and the kernel spills (540 bytes of reloads, 1032 with parameterised
// gates); without, 340 and 436.  64 instances of 20 qubits 2.01 -> 1.87 ms,
// eight of 23 2.16 -> 1.97 ms (lockstep rounds: 1.88 and 1.98).  Resident
// CTAs per SM of each (occupancy API, set by batch_wide_setup before any
// launch or capture).
static decltype(&k_batch_persistent_wide<false, 2>) const g_wide_kern[2][2] = {
    {k_batch_persistent_wide<false, 2>, k_batch_persistent_wide<false, 1>},
    {k_batch_persistent_wide<true, 2>, k_batch_persistent_wide<true, 1>}};
static int g_wide_per_sm[2][2] = {{3, 3}, {3, 3}};

qs_status launch_batch_persistent_wide(cudaStream_t st, int num_sms, void *amps, const PersistItem *items, int nitems,
                                       const WidePass *passes, const WideOp *ops, const uint8_t *codes,
                                       const FoldArgs *folds, uint32_t *done, PersistCtl *ctl, double *part,
                                       double *sums, bool any_full, bool grouped)
{
    if (nitems <= 0) return QS_OK;
    const int cap = num_sms * g_wide_per_sm[any_full][grouped];
    g_wide_kern[any_full][grouped]<<<nitems < cap ? nitems : cap, kWideThreads, 65536, st>>>(
        (float2 *)amps, items, nitems, passes, ops, codes, folds, done, ctl, part, sums, kPersistWaitNs);
    QS_LAUNCH_CHECK();
    return QS_OK;
}

qs_status batch_wide_setup()
{
    const int dyn = 65536;
    QS_CUDA_TRY(cudaFuncSetAttribute(k_batch_pass_wide<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn));
    QS_CUDA_TRY(cudaFuncSetAttribute(k_batch_pass_wide<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn));
    for (int f = 0; f < 2; ++f)
        for (int g = 0; g < 2; ++g) {
            QS_CUDA_TRY(cudaFuncSetAttribute(g_wide_kern[f][g], cudaFuncAttributeMaxDynamicSharedMemorySize, dyn));
            int &v = g_wide_per_sm[f][g];
            QS_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, g_wide_kern[f][g], kWideThreads, dyn));
            v = v < 1 ? 1 : v;
        }
    return QS_OK;
}

QS_CHECK_READER(check_poll_wide)

}  // namespace qs
