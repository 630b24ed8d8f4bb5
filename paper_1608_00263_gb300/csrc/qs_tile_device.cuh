// qs_tile_device.cuh -- device helpers shared by the fused tile passes: the
// shared-memory swizzle, the register slots' loads and stores, and index
// deposits.
#pragma once

#include "qs_device.cuh"

namespace qs {

// Swizzled shared-memory index of tile element e: elements are grouped in
// 16-byte units u = e / CE; bits 0..2 of u are XORed with a fold of its
// higher bits.  Linear over GF(2): swz(a ^ b) = swz(a) ^ swz(b).
template <int CE>
__host__ __device__ __forceinline__ uint32_t swz(uint32_t e)
{
    return tile_swizzle(e, CE);
}

// Trailing zeros of a positive integer known at compile time (the callers
// use it on unrolled loop indices, so it folds to a constant).
template <int X> struct CtzT { static constexpr int value = (X & 1) ? 0 : 1 + CtzT<(X >> 1)>::value; };
template <> struct CtzT<0> { static constexpr int value = 0; };

// Loads / stores the register slots of a phase from / to the shared tile,
// visiting slots in Gray-code order so that each address differs from the
// previous one by one register bit (one XOR with that bit's offset); the two
// halves of the slots run as two interleaved chains.
// COUNT slots (or slot pairs when SHIFT = 1: register bit 0 is tile bit 0,
// so slots s and s+1 are one 16-byte unit).
template <int COUNT, int SHIFT>
struct SlotIO {
    // offsets are in bytes from the start of the tile
    // two Gray-code chains, one per half of the slots (top register bit
    // clear / set): half the dependent address XORs per load sequence
    static constexpr int kTop = CtzT<COUNT>::value - 1;
    template <int I, typename V>
    struct Step2 {
        static __device__ __forceinline__ void ld(V *a, const char *tile, uint32_t o0, uint32_t o1, const uint32_t *pb)
        {
            if (I) { o0 ^= pb[SHIFT + CtzT<I>::value]; o1 ^= pb[SHIFT + CtzT<I>::value]; }
            constexpr int s0 = (I ^ (I >> 1)) << SHIFT;
            constexpr int s1 = s0 + ((COUNT / 2) << SHIFT);
            if (SHIFT) {
                const float4 v = *reinterpret_cast<const float4 *>(tile + o0);
                const float4 w = *reinterpret_cast<const float4 *>(tile + o1);
                a[s0].x = v.x; a[s0].y = v.y; a[s0 + 1].x = v.z; a[s0 + 1].y = v.w;
                a[s1].x = w.x; a[s1].y = w.y; a[s1 + 1].x = w.z; a[s1 + 1].y = w.w;
            } else {
                a[s0] = *reinterpret_cast<const V *>(tile + o0);
                a[s1] = *reinterpret_cast<const V *>(tile + o1);
            }
            Step2<I + 1, V>::ld(a, tile, o0, o1, pb);
        }
        static __device__ __forceinline__ void st(const V *a, char *tile, uint32_t o0, uint32_t o1, const uint32_t *pb)
        {
            if (I) { o0 ^= pb[SHIFT + CtzT<I>::value]; o1 ^= pb[SHIFT + CtzT<I>::value]; }
            constexpr int s0 = (I ^ (I >> 1)) << SHIFT;
            constexpr int s1 = s0 + ((COUNT / 2) << SHIFT);
            if (SHIFT) {
                *reinterpret_cast<float4 *>(tile + o0) = make_float4(a[s0].x, a[s0].y, a[s0 + 1].x, a[s0 + 1].y);
                *reinterpret_cast<float4 *>(tile + o1) = make_float4(a[s1].x, a[s1].y, a[s1 + 1].x, a[s1 + 1].y);
            } else {
                *reinterpret_cast<V *>(tile + o0) = a[s0];
                *reinterpret_cast<V *>(tile + o1) = a[s1];
            }
            Step2<I + 1, V>::st(a, tile, o0, o1, pb);
        }
    };
    template <typename V>
    struct Step2<COUNT / 2, V> {
        static __device__ __forceinline__ void ld(V *, const char *, uint32_t, uint32_t, const uint32_t *) {}
        static __device__ __forceinline__ void st(const V *, char *, uint32_t, uint32_t, const uint32_t *) {}
    };
    template <typename V>
    static __device__ __forceinline__ void load(V *a, const char *tile, uint32_t off, const uint32_t *pb)
    { Step2<0, V>::ld(a, tile, off, off ^ pb[SHIFT + kTop], pb); }
    template <typename V>
    static __device__ __forceinline__ void store(const V *a, char *tile, uint32_t off, const uint32_t *pb)
    { Step2<0, V>::st(a, tile, off, off ^ pb[SHIFT + kTop], pb); }
};

// Deposits the low bits of x into the positions listed in pos[0..cnt).
__device__ __forceinline__ uint64_t deposit(uint64_t x, const uint8_t *pos, int cnt)
{
    uint64_t r = 0;
    for (int i = 0; i < cnt; ++i) r |= ((x >> i) & 1ULL) << pos[i];
    return r;
}

__device__ __forceinline__ uint32_t smem_addr(const void *p)
{
    return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mul_sign(float2 &v, float sg) { v = __fmul2_rn(v, make_float2(sg, sg)); }
__device__ __forceinline__ void mul_sign(double2 &v, double sg) { v.x *= sg; v.y *= sg; }

// complex64 slot <-> 64-bit word (re in the low half) for the PTX op loop
__device__ __forceinline__ unsigned long long f2_bits(float2 v)
{
    return ((unsigned long long)__float_as_uint(v.y) << 32) | __float_as_uint(v.x);
}
__device__ __forceinline__ float2 bits_f2(unsigned long long b)
{
    return make_float2(__uint_as_float((uint32_t)b), __uint_as_float((uint32_t)(b >> 32)));
}

}  // namespace qs
