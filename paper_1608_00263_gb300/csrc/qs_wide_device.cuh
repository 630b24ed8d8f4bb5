// qs_wide_device.cuh -- body of the wide fused pass (complex64).
//
// The same tile pass as in qs_fused.cu -- a tile of 2^t amplitudes in shared
// memory, register phases, one byte code per op -- with 64 amplitudes (6
// register bits) per thread instead of 32, held as packed pairs of real and
// of imaginary parts (gen_op_loop.py).  The pass is bound by instruction
// issue and by the latency of its op dispatch, not by HBM, so what counts is
// the work per issued instruction: every gate outside register bit 0 is
// packed FP32x2 arithmetic (X^1/2 and T half the instructions of the
// (re, im) layout), and twice the amplitudes per thread halve dispatch,
// addressing and tables.  Register bit 0 is tile bit 0 in every phase, so all
// slot accesses are 16 bytes.  128 threads hold a 13-qubit tile at 168
// registers and 75 KB of shared memory, so three CTAs share an SM: while one
// waits for its tile, two compute.
//
// A state of few tiles has one or two CTAs per SM, one or two warps per
// scheduler, and every latency shows (12 qubits: an instruction in 5 cycles,
// waiting in turn for shared memory, fixed latencies and instruction fetch):
// there 32 amplitudes (5 register bits) per thread and twice the warps are
// the better split (RB = 5; rule and figures in default_plan_params).
#pragma once

#include <cstddef>

#include "qs_tile_device.cuh"

namespace qs {

#include "qs_op_loop.inc"

constexpr int kWideThreads = 1 << (13 - kWideRegBits);   // threads of a 13-qubit tile
constexpr int kWideSlots = 1 << kWideRegBits;

constexpr uint32_t kWideDirect = 4, kWideMore = 8, kWideCanon = 16;   // phase flags (gen_op_loop.py)

struct alignas(16) WideUnit {           // unit `it` of every thread
    uint64_t goff;          // byte offset in the state
    uint32_t soff;          // swizzled byte offset in the tile
    uint32_t pad;
};

template <int RB>
struct WideSmemT {
    static constexpr int kThreads = 1 << (13 - RB), kUnits = 1 << (RB - 1);   // 16-byte units per thread
    WidePass P;
    WideOp ops[kMaxWideOps];
    uint32_t codes[kMaxWideOps / 4 + 4];
    uint64_t toff[kThreads];                     // byte offset in the state of the thread's first copied unit
    uint64_t doff[kThreads];                     // ... of its slot 0 in the last phase
    uint64_t dst[kThreads];                      // state address of the thread's slot 0 of this tile
    uint64_t amps;                                   // the state, and the end of the tile range: read
    uint32_t t_end, pad;                             // again where used, registers are short
    alignas(16) uint64_t part;                       // adjoint sweep: partials of this CTA's warps,
    uint64_t part_stride;                            // bytes per slot
    uint64_t gmask;                                  // out-of-tile qubits
    uint16_t thr[kMaxPhasesPerPass][kThreads];   // tile element of the thread's slot 0
    WideUnit unit[kUnits];
    float2 w8[8];                                    // e^{i pi k / 4}
};

using WideSmem = WideSmemT<kWideRegBits>;

static_assert(sizeof(WidePass) % 16 == 0 && offsetof(WidePass, ph) % 16 == 0 && offsetof(WideSmem, ops) % 16 == 0 &&
                  offsetof(WideSmem, unit) % 16 == 0 && offsetof(WideSmem, part) % 16 == 0 && sizeof(WideUnit) == 16,
              "staged in 16-byte units");

// Tables of the folded diagonal prefix (first pass of a circuit, see
// FoldArgs): CZ partners as a qubit mask and as a mask of tile bits, T
// counts, the unit table, and 2^(-n/2) e^{i pi k / 4}.
struct WideFoldSmem {
    uint64_t nb[kMaxQubits];
    uint64_t m[3];
    uint32_t plain;         // nothing folded: every amplitude is 2^(-n/2) (FOLD 1)
    uint16_t g[kMaxQubits];
    uint8_t u[kWideSlots];
    float2 w[8];
};

// A unit between canonical order (re, im, re, im) and (re, re, im, im).
__device__ __forceinline__ float4 swap_unit(float4 v) { return make_float4(v.x, v.z, v.y, v.w); }

// Barrier of a tile's threads: the CTA, or its group of whole warps.
template <int GROUPED>
__device__ __forceinline__ void wide_sync(int nthr, int gi)
{
    if constexpr (GROUPED == 0) __syncthreads();
    else asm volatile("bar.sync %0, %1;" ::"r"(gi + 1), "r"(nthr) : "memory");
}

// Runs tiles [t_begin, t_end) of one pass on `amps`.  blockDim.x threads; a
// tile takes 2^(t - 6) of them: all (GROUPED 0), a group of whole warps (t >=
// 11) with its own tile buffer, group g running tiles t_begin + g, + groups,
// ... (GROUPED 1), or the first ones, the others idle (GROUPED 2: fewer
// registers than groups; for passes of one small tile).
// FOLD 1: a circuit's first pass, which writes its tiles
// (the uniform state times the folded prefix's phases) instead of loading
// them; F's nb and m are set by the caller (published by the first barrier).
// FOLD 2: the same where the pass says so (its prefix in folds_g).
// The caller's CTA is converged; ends with a CTA barrier.
// KIND: the op loop (0 Clifford+T, 1 all gates, 2 the adjoint sweep, whose
// tile bit t - 1 selects psi or lambda, lam_off bytes away; S.part and
// S.part_stride are set by the caller).
template <int KIND, int FOLD, int GROUPED, int RB = kWideRegBits>
__device__ __forceinline__ void wide_pass_body(float2 *__restrict__ amps, const WidePass *__restrict__ pass_g,
                                               const WideOp *__restrict__ ops_g, const uint8_t *__restrict__ codes_g,
                                               uint32_t t_begin, uint32_t t_end, WideSmemT<RB> &S, WideFoldSmem *F,
                                               unsigned char *smem_raw, uint64_t lam_off = 0,
                                               const FoldArgs *__restrict__ folds_g = nullptr)
{
    using Smem = WideSmemT<RB>;
    constexpr int NS = 1 << RB, NU = NS / 2;
    for (int i = threadIdx.x; i < (int)(sizeof(WidePass) / 4); i += blockDim.x)
        reinterpret_cast<uint32_t *>(&S.P)[i] = reinterpret_cast<const uint32_t *>(pass_g)[i];
    __syncthreads();
    const int t = S.P.t, ng = S.P.n - t, nph = S.P.nphases, nops = S.P.nops;
    // whether the tiles are generated
    auto gen = [&]() { return FOLD == 1 || (FOLD == 2 && S.P.fold != 0); };
    if constexpr (FOLD == 2) {
        if (S.P.fold) {
            const FoldArgs &f = folds_g[S.P.fold - 1];
            for (int i = threadIdx.x; i < kMaxQubits; i += blockDim.x) F->nb[i] = f.nb[i];
            if (threadIdx.x == 0) {
                F->m[0] = f.m1;
                F->m[1] = f.m2;
                F->m[2] = f.m4;
            }
            __syncthreads();
        }
    }
    const int nthr = GROUPED ? 1 << (t - RB) : (int)blockDim.x;
    const int tid = GROUPED == 1 ? (int)(threadIdx.x & (unsigned)(nthr - 1)) : (int)threadIdx.x;
    const int gi = GROUPED == 1 ? (int)(threadIdx.x >> (t - RB)) : 0;
    const int ngr = GROUPED == 1 ? (int)(blockDim.x >> (t - RB)) : 1;
    const bool idle = GROUPED == 2 && (int)threadIdx.x >= nthr;
    // byte offset in the state of tile element e
    auto state_off = [&](uint32_t e) -> uint64_t {
        if constexpr (KIND == 2)
            return deposit(e & ((1u << (t - 1)) - 1u), S.P.L, t - 1) * 8u + ((e >> (t - 1)) & 1u ? lam_off : 0ull);
        else
            return deposit(e, S.P.L, t) * 8u;
    };
    // ---- stage the ops and the per-thread tables (once per CTA and pass) ----
    {
        const uint4 *src = reinterpret_cast<const uint4 *>(ops_g + S.P.op_begin);
        for (int i = threadIdx.x; i < nops; i += blockDim.x) reinterpret_cast<uint4 *>(S.ops)[i] = src[i];
        const uint32_t *cw = reinterpret_cast<const uint32_t *>(codes_g + S.P.op_begin);
        for (int i = threadIdx.x; i < (nops + 7) / 4; i += blockDim.x) S.codes[i] = cw[i];
    }
    if (gi == 0 && !idle)
        for (int ph = 0; ph < nph; ++ph) {
            uint32_t e = 0;
            for (int k = 0; k < t - RB; ++k) e |= (((uint32_t)tid >> k) & 1u) << S.P.ph[ph].T[k];
            S.thr[ph][tid] = (uint16_t)e;
        }
    for (int i = threadIdx.x; i < NU; i += blockDim.x) {
        const uint32_t e = 2u * (uint32_t)nthr * (uint32_t)i;
        S.unit[i].goff = state_off(e);
        S.unit[i].soff = swz<2>(e) * 8u;
    }
    if (threadIdx.x < 8) {
        const float c = 0.70710678118654752440f;
        const int k = (int)threadIdx.x;
        const float re = (k & 3) == 2 ? 0.f : (k & 3) == 0 ? 1.f : ((k & 3) == 1 ? c : -c);
        const float im = (k & 3) == 0 ? 0.f : (k & 3) == 2 ? 1.f : c;
        S.w8[k] = k < 4 ? make_float2(re, im) : make_float2(-re, -im);
    }
    auto fcount = [&](int q) -> uint32_t {
        return (uint32_t)((F->m[0] >> q) & 1) + 2u * (uint32_t)((F->m[1] >> q) & 1) + 4u * (uint32_t)((F->m[2] >> q) & 1);
    };
    if (FOLD && gen() && !(FOLD == 1 && F->plain)) {
        // each qubit's CZ partners as tile bits
        for (int q = threadIdx.x; q < S.P.n; q += blockDim.x) {
            uint32_t m = 0;
            for (int b = 0; b < t; ++b) m |= (uint32_t)((F->nb[q] >> S.P.L[b]) & 1) << b;
            F->g[q] = (uint16_t)m;
        }
        // unit u = (it, q) of every thread: tile element 2 nthr it + q;
        // 4 (CZ pairs among its tile bits) + (its T counts), mod 8
        for (int u = threadIdx.x; u < NS; u += blockDim.x) {
            const uint32_t eu = 2u * (uint32_t)nthr * (uint32_t)(u / 2) + (uint32_t)(u & 1);
            uint32_t pairs = 0, tcnt = 0;
            for (uint32_t w = eu; w; w &= w - 1) {
                const int qb = S.P.L[__ffs(w) - 1];
                for (uint32_t v = w & (w - 1); v; v &= v - 1) pairs += (uint32_t)(F->nb[qb] >> S.P.L[__ffs(v) - 1]) & 1u;
                tcnt += fcount(qb);
            }
            F->u[u] = (uint8_t)((4u * (pairs & 1u) + tcnt) & 7u);
        }
    }
    if (FOLD && gen() && threadIdx.x < 8) {
        // 2^(-n/2) e^{i pi k / 4}: both factors of 2^(-n/2) are exact but for
        // the rounding of 1/sqrt2
        const int k = (int)threadIdx.x;
        const double s = 0.70710678118654752440;
        const double a = __hiloint2double((1023 - (S.P.n >> 1)) << 20, 0) * (S.P.n & 1 ? s : 1.0), c = a * s;
        const double re = (k & 3) == 2 ? 0.0 : (k & 3) == 0 ? a : ((k & 3) == 1 ? c : -c);
        const double im = (k & 3) == 0 ? 0.0 : (k & 3) == 2 ? a : c;
        F->w[k] = k < 4 ? make_float2((float)re, (float)im) : make_float2((float)-re, (float)-im);
    }
    if (gi == 0 && !idle) {
        S.toff[tid] = state_off(2u * (uint32_t)tid);
        S.doff[tid] = state_off(S.thr[nph - 1][tid]);
    }
    if (threadIdx.x == 0) {
        uint64_t m = 0;
        for (int i = 0; i < ng; ++i) m |= 1ULL << S.P.G[i];
        S.gmask = m;
        S.amps = reinterpret_cast<uint64_t>(amps);
        S.t_end = t_end;
        if constexpr (KIND == 2) S.P.dreg[RB - 1] = lam_off;
    }
    __syncthreads();
    unsigned char *gsm = GROUPED == 1 ? smem_raw + (((size_t)gi << t) * sizeof(float2)) : smem_raw;
    const uint32_t tile_sa = smem_addr(gsm);
    const uint32_t sw_tid = swz<2>(2u * (uint32_t)tid) * 8u;
    uint32_t tau = idle ? t_end : t_begin + (uint32_t)gi;
    uint64_t base = deposit(tau, S.P.G, ng);
    // the tile's highest element index must lie inside the state
    auto inside = [&](uint64_t b) {
        uint64_t lmask = 0;
#ifdef QS_CHECKED
        for (int i = 0; i < t; ++i) lmask |= 1ULL << S.P.L[i];
#endif
        (void)lmask;
        (void)b;
        return QS_DCHECK(((b | lmask) >> S.P.n) == 0, 202);
    };
    if (!gen()) {
        if (tau < S.t_end && inside(base)) {
            const char *src = reinterpret_cast<const char *>(amps) + (base * 8u + S.toff[tid]);
#pragma unroll 4
            for (int it = 0; it < NU; ++it)
                asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(tile_sa + (sw_tid ^ S.unit[it].soff)),
                             "l"(src + S.unit[it].goff)
                             : "memory");
        }
    }
    while (tau < S.t_end && inside(base)) {
        S.dst[threadIdx.x] = S.amps + base * 8u + S.doff[tid];
        if (FOLD == 1 && F->plain) {
            // (28 qubits, the layer and one R_X: 438 us; 619 with every
            // element's phase formed from empty masks)
            const float2 w = F->w[0];
#pragma unroll 4
            for (int it = 0; it < NU; ++it)
                *reinterpret_cast<float4 *>(gsm + (sw_tid ^ S.unit[it].soff)) = make_float4(w.x, w.x, w.y, w.y);
        } else if (FOLD && gen()) {
            // element x gets 2^(-n/2) e^{i pi k(x) / 4}, k = 4 (CZ pairs within
            // x) + (T counts of x), mod 8, summed over the out-of-tile bits,
            // the thread's tile bits and the unit's, plus the pairs across
            uint32_t pb = 0, nbm = 0;
            for (uint64_t w = base; w; w &= w - 1) {
                const int i = __ffsll((long long)w) - 1;
                pb ^= (uint32_t)__popcll(base & F->nb[i] & (~0ULL << i << 1));
                nbm ^= F->g[i];
            }
            const uint32_t lb = (uint32_t)(__popcll(base & F->m[0]) + 2 * __popcll(base & F->m[1]) +
                                           4 * __popcll(base & F->m[2]));
            const uint32_t et = 2u * (uint32_t)tid;
            uint32_t pt = 0, nt = 0, lt = 0;
            for (uint32_t w = et; w; w &= w - 1) {
                const int b = __ffs(w) - 1;
                const int q = S.P.L[b];
                pt ^= (uint32_t)__popc(et & (uint32_t)F->g[q] & (~0u << b << 1));
                nt ^= F->g[q];
                lt += fcount(q);
            }
            const uint32_t k0 = 4u * ((pb ^ pt ^ (uint32_t)__popc(et & nbm)) & 1u) + lb + lt;
            const uint32_t nu = nbm ^ nt;
#pragma unroll 4
            for (int it = 0; it < NU; ++it) {
                float2 fill[2];
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const uint32_t eu = 2u * (uint32_t)nthr * (uint32_t)it + (uint32_t)q;
                    fill[q] = F->w[(k0 + F->u[it * 2 + q] + 4u * ((uint32_t)__popc(eu & nu) & 1u)) & 7u];
                }
                *reinterpret_cast<float4 *>(gsm + (sw_tid ^ S.unit[it].soff)) =
                    make_float4(fill[0].x, fill[1].x, fill[0].y, fill[1].y);
            }
        }
        asm volatile("cp.async.wait_all;\n" ::: "memory");
        if (FOLD != 1 && S.P.canon_in) {
            // the units this thread copied, to the order the phases work on
#pragma unroll 4
            for (int it = 0; it < NU; ++it) {
                float4 *u = reinterpret_cast<float4 *>(gsm + (sw_tid ^ S.unit[it].soff));
                *u = swap_unit(*u);
            }
        }
        wide_sync<GROUPED>(nthr, gi);
        // (this tile's base is read back from the thread's address, and the
        // next one formed, where they are used)
        auto this_base = [&]() { return (S.dst[threadIdx.x] - S.amps - S.doff[tid]) >> 3; };
        auto next_base = [&]() {
            return GROUPED == 1 && ngr > 1 ? deposit(tau + (uint32_t)ngr, S.P.G, ng)
                                      : (((this_base() | ~S.gmask) + 1) & S.gmask);
        };
        for (int ph = 0; ph < nph; ++ph) {
            const WidePhase &H = S.P.ph[ph];
            const uint32_t te = S.thr[ph][tid], to = tau;
            const int ub = H.tail_begin, oe = H.op_end;
            // diagonal ops selected outside the register set scale the
            // thread's slots by one factor: T and sign flips count eighths
            // of a turn (their codes), general phases multiply; the last
            // phase adds the pass-wide factor
            const bool last = ph == nph - 1;
            float fr = 1.f, fi = 0.f;
            uint32_t mode = 0;
            if (ub < oe || last) {
                uint32_t k = 0;
#pragma unroll 2
                for (int o = ub; o < oe; ++o) {
                    const WideOp op = S.ops[o];
                    if ((te & op.sel_tile) == op.sel_tile && (to & op.sel_out) == op.sel_out) {
                        k += reinterpret_cast<const uint8_t *>(S.codes)[o];
                        if constexpr (KIND > 0) {
                            const float x = fr * op.p0 - fi * op.p1;
                            fi = fr * op.p1 + fi * op.p0;
                            fr = x;
                        }
                    }
                }
                const float2 w = S.w8[k & 7u];
                float x = fr * w.x - fi * w.y;
                fi = fr * w.y + fi * w.x;
                fr = x;
                if (last) {
                    const float gr = S.P.gs_re, gim = S.P.gs_im;
                    x = fr * gr - fi * gim;
                    fi = fr * gim + fi * gr;
                    fr = x;
                }
                mode = __any_sync(0xffffffffu, fi != 0.f) ? 2u : 1u;
            }
            const bool direct = last && S.P.direct;
            const char *nsrc = nullptr;
            if (direct) {
                mode |= kWideDirect | (S.P.canon_out ? kWideCanon : 0u);
                const uint64_t nbase = next_base();
                if (!gen() && tau + (uint32_t)ngr < S.t_end && inside(nbase)) {
                    mode |= kWideMore;
                    nsrc = reinterpret_cast<const char *>(S.amps + (nbase * 8u + S.toff[tid]));
                }
            }
            OpLoop<KIND, RB>::template run<(int)offsetof(Smem, codes), (int)offsetof(Smem, ops) - 16,
                                           (int)offsetof(Smem, unit),
                                           (int)(offsetof(Smem, P) + offsetof(WidePass, dreg)),
                                           (int)offsetof(Smem, dst), (int)offsetof(Smem, part)>(
                swz<2>(te) * 8u, tile_sa, smem_addr(&S),
                (uint32_t)(offsetof(Smem, P) + offsetof(WidePass, ph)) + (uint32_t)ph * (uint32_t)sizeof(WidePhase),
                H.op_begin, ((uint64_t)to << 32) | te, fr, fi, mode, sw_tid,
                nsrc, GROUPED ? (uint32_t)gi + 1u : 0u,
                (uint32_t)nthr);
            if (!direct) wide_sync<GROUPED>(nthr, gi);
        }
        // ---- staged pass: store the tile; each unit's place takes the same
        // unit of the next tile as soon as this thread has read it (no other
        // thread touches it before the next barrier) ----
        if (!S.P.direct) {
            const uint64_t toff = S.toff[tid], nbase = next_base();
            const bool more = !gen() && tau + (uint32_t)ngr < S.t_end && inside(nbase), canon_out = S.P.canon_out != 0;
            char *dst = reinterpret_cast<char *>(S.amps + (this_base() * 8u + toff));
            const char *src = reinterpret_cast<const char *>(S.amps + (nbase * 8u + toff));
#pragma unroll 4
            for (int i0 = 0; i0 < NU; i0 += 2) {
                WideUnit u[2];
                float4 v[2];
#pragma unroll
                for (int i = 0; i < 2; ++i) {
                    u[i] = S.unit[i0 + i];
                    u[i].soff ^= sw_tid;
                }
#pragma unroll
                for (int i = 0; i < 2; ++i) v[i] = *reinterpret_cast<const float4 *>(gsm + u[i].soff);
#pragma unroll
                for (int i = 0; i < 2; ++i)
                    *reinterpret_cast<float4 *>(dst + u[i].goff) = canon_out ? swap_unit(v[i]) : v[i];
                if (more) {
#pragma unroll
                    for (int i = 0; i < 2; ++i)
                        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(tile_sa + u[i].soff),
                                     "l"(src + u[i].goff)
                                     : "memory");
                }
            }
        }
        base = next_base();
        tau += (uint32_t)ngr;
    }
    __syncthreads();
}

}  // namespace qs
