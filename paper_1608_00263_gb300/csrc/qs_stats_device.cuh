// qs_stats_device.cuh -- device helpers of the output statistics: the
// per-element terms of the Porter-Thomas statistics and the fixed-order
// block reduction, shared by the single-state read-out, the batched
// statistics kernels and the persistent ensemble kernel.
#pragma once

#include "qs_device.cuh"

namespace qs {

constexpr int kStatThreads = 256;
constexpr int kStatAcc = 12;   // sum y, sum y ln y, sum ln y, sum y^k (k=2..10)

// ---------------------------------------------------------------------------
// block reduction helpers (fixed order)
// ---------------------------------------------------------------------------
__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Sums acc[k] over the warp for every k < K <= 16 by recursive halving: at
// each step a lane hands half of its sums to its partner and keeps the other
// half, so a warp spends K (rounded up to 16) additions in all instead of
// 5 K.  FP64 additions are what bounds this tail (two lanes per clock and
// SM).  Lane l returns the total of accumulator (l & 15) (K <= l: 0).
template <int K>
__device__ __forceinline__ double warp_sum_many(const double (&acc)[K])
{
    static_assert(K <= 16, "at most 16 accumulators");
    const int lane = threadIdx.x & 31;
    double v[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = k < K ? acc[k < K ? k : 0] : 0.0;
    // bit o of the lane selects the upper half of the sums left
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) {
        const bool up = (lane & o) != 0;
#pragma unroll
        for (int k = 0; k < o; ++k) {
            const double give = up ? v[k] : v[k + o], keep = up ? v[k + o] : v[k];
            v[k] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
    return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 16);
}

// Sums acc over the block's THREADS threads (recursive halving inside a
// warp, then the warps' sums in warp order) and stores the K sums at dst
// (threads < K).
template <int K, int THREADS = kStatThreads>
__device__ __forceinline__ void block_sum_store(double (&acc)[K], double *dst)
{
    __shared__ double red[THREADS / 32][16];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if constexpr (K >= 4) {
        const double v = warp_sum_many<K>(acc);
        if (lane < 16) red[warp][lane] = v;
    } else {
#pragma unroll
        for (int k = 0; k < K; ++k) {
            const double v = warp_sum(acc[k]);
            if (lane == 0) red[warp][k] = v;
        }
    }
    __syncthreads();
    if (threadIdx.x < K) {
        double s = 0;
        for (int w = 0; w < THREADS / 32; ++w) s += red[w][threadIdx.x];
        dst[threadIdx.x] = s;
    }
}

// Accumulates one element's contributions.  y = N p.
template <typename T>
__device__ __forceinline__ void stat_terms(T y, T (&c)[kStatAcc])
{
    T ly = (sizeof(T) == 4) ? (T)__logf((float)y) : (T)log((double)y);
    c[0] += y;
    c[1] += (y > (T)0) ? y * ly : (T)0;
    c[2] += ly;
    T yk = y;
#pragma unroll
    for (int k = 2; k <= 10; ++k) {
        yk *= y;
        c[k + 1] += yk;
    }
}

// Statistics partials of one chunk of a complex64 state (cnt amplitudes at
// a, cnt even, a 16-byte aligned; scaleN = N of the instance): each thread
// takes 16-byte pairs of amplitudes blockDim.x apart, eight loads in flight
// at a time, and sums the terms of 64 amplitudes in FP32 before adding them
// into FP64 accumulators (terms of y = N p > 4096 formed in FP64); then the
// block's fixed-order sum goes to dst[0 .. kStatAcc).  The whole block
// (THREADS threads) calls it.  Amplitudes are read through L2
// (ld.global.cg), so the chunk may have been written earlier in the same
// launch by another CTA (after an acquire of that CTA's release).
// BATCHED: one test per sixteen amplitudes, so that their logarithms and powers
// overlap (with a branch at each, one chain runs after the other): for few warps
// per SM, where nothing else hides the chains.  It takes 158 registers instead
// of 122; with many CTAs per SM to hide them the plain form wins.  The same sums
// either way.
template <int THREADS = kStatThreads, bool BATCHED = false>
__device__ __forceinline__ void batch_stats_chunk(const float2 *a, uint64_t cnt, float scaleN, double *dst)
{
    constexpr int kLoads = 8;                      // 16-byte loads in flight per thread
    constexpr int kGroup = 32;                     // pairs per FP32 partial (64 amplitudes)
    const float4 *a4 = reinterpret_cast<const float4 *>(a);
    const uint64_t units = cnt / 2, bd = blockDim.x;
    double acc[kStatAcc];
#pragma unroll
    for (int k = 0; k < kStatAcc; ++k) acc[k] = 0;
    for (uint64_t u0 = threadIdx.x; u0 < units; u0 += bd * kGroup) {
        float c[kStatAcc];
#pragma unroll
        for (int k = 0; k < kStatAcc; ++k) c[k] = 0.f;
        for (int j0 = 0; j0 < kGroup; j0 += kLoads) {
            float4 v[kLoads];
#pragma unroll
            for (int k = 0; k < kLoads; ++k) {
                const uint64_t u = u0 + (uint64_t)(j0 + k) * bd;
                v[k] = u < units ? __ldcg(a4 + u) : make_float4(0.f, 0.f, 0.f, 0.f);
            }
            if constexpr (BATCHED) {
                float y[2 * kLoads], top = 0.f;
#pragma unroll
                for (int k = 0; k < kLoads; ++k) {
                    y[2 * k] = (v[k].x * v[k].x + v[k].y * v[k].y) * scaleN;
                    y[2 * k + 1] = (v[k].z * v[k].z + v[k].w * v[k].w) * scaleN;
                    top = fmaxf(top, fmaxf(y[2 * k], y[2 * k + 1]));
                }
                if (top <= 4096.f && u0 + (uint64_t)(j0 + kLoads - 1) * bd < units) {
#pragma unroll
                    for (int k = 0; k < 2 * kLoads; ++k) stat_terms<float>(y[k], c);
                    continue;
                }
            }
#pragma unroll
            for (int k = 0; k < kLoads; ++k) {
                if (u0 + (uint64_t)(j0 + k) * bd >= units) continue;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const float re = h ? v[k].z : v[k].x, im = h ? v[k].w : v[k].y;
                    const float y = (re * re + im * im) * scaleN;
                    if (y > 4096.f) stat_terms<double>(((double)re * re + (double)im * im) * (double)scaleN, acc);
                    else stat_terms<float>(y, c);
                }
            }
        }
#pragma unroll
        for (int k = 0; k < kStatAcc; ++k) acc[k] += (double)c[k];
    }
    block_sum_store<kStatAcc, THREADS>(acc, dst);
}

}  // namespace qs
