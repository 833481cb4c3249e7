// heget_reduce.cuh -- combination of Monte Carlo partials (double-double sums
// and counters) across the threads of a block and across blocks.
//
// Partials are combined in integers: every term is aligned to the largest
// exponent among them as a 128-bit fixed-point number, the numbers are added
// as integers, and the total goes back to a double-double.  The additions are
// exact, so the result does not depend on their order; what is lost are bits
// below 2^-113 (a block) or 2^-(124 - log2 terms) (a whole grid) of the largest
// term, below the 2^-104 of a double-double addition.
//
// Why integers: GB300 issues a warp's FP64 instruction in 64 cycles of its
// sub-partition whatever the number of active lanes, and a double-double
// addition takes 20 of them.  A tree of double-double additions over a
// 256-thread block (5 shuffle levels x 2 sums, then 7 by one thread) held the
// FP64 pipe at the end of every block -- 600 of the 1160 FP64 instructions a
// point of a 128-point FP64 tile at n = 2 -- and the one-block finalisation
// for 43 us.  The integer form is about 300 integer instructions a warp.
// GB300, before -> after: one call of 1000 points at n = 2 102 -> 41 us, 65,536
// points in FP64 228 -> 96 us, n = 4 FP32 1,048,576 points 1202 -> 1123 us, FP64
// 262,144 points 3483 -> 3030 us, a batch of 24 mixed requests 4883 -> 4286 us,
// with the same bits in every result.  (The gain of this form alone; with the
// ones that followed these calls take 33, 66, 611, 1587 and 3212 us.)
#pragma once

#include "heget_common.cuh"

namespace heget {

__host__ __device__ __forceinline__ unsigned long long double_bits(double x) {
#ifdef __CUDA_ARCH__
    return (unsigned long long)__double_as_longlong(x);
#else
    unsigned long long u;
    __builtin_memcpy(&u, &x, sizeof u);
    return u;
#endif
}
__host__ __device__ __forceinline__ double bits_double(unsigned long long u) {
#ifdef __CUDA_ARCH__
    return __longlong_as_double((long long)u);
#else
    double x;
    __builtin_memcpy(&x, &u, sizeof x);
    return x;
#endif
}

// Biased exponent of x, 1 for zero and subnormals, 0x7FF for inf and NaN.
__host__ __device__ __forceinline__ int exponent_field(double x) {
    const int e = (int)(double_bits(x) >> 52) & 0x7FF;
    return e > 0 ? e : 1;
}
__host__ __device__ __forceinline__ int exponent_field(const DD& a) {
    const int h = exponent_field(a.hi), l = exponent_field(a.lo);
    return h > l ? h : l;
}

// x as an integer in units of 2^(em - 1075 - top), truncated towards zero;
// em >= the exponent field of x, 0 <= top <= 73.  A term is below
// 2^(53 + top) in magnitude: up to 2^(73 - top) of them add up without
// overflow.
__host__ __device__ __forceinline__ __int128 fixed_of(double x, int em, int top) {
    const unsigned long long u = double_bits(x);
    const int ef = (int)(u >> 52) & 0x7FF;
    unsigned long long m = u & 0xFFFFFFFFFFFFFull;
    if (ef) m |= 1ull << 52;
    const int sh = top - (em - (ef ? ef : 1));
    unsigned __int128 v = m;
    if (sh >= 0) v <<= sh;
    else v = sh > -64 ? (unsigned __int128)(m >> -sh) : 0;
    return (u >> 63) ? -(__int128)v : (__int128)v;
}
__host__ __device__ __forceinline__ __int128 fixed_of(const DD& a, int em, int top) {
    return fixed_of(a.hi, em, top) + fixed_of(a.lo, em, top);
}

__host__ __device__ __forceinline__ int clz64(unsigned long long x) {
#ifdef __CUDA_ARCH__
    return __clzll((long long)x);
#else
    return x ? __builtin_clzll(x) : 64;
#endif
}

// m 2^e (m < 2^53) as a double, exact unless it leaves the double range.
__host__ __device__ __forceinline__ double scaled_int(unsigned long long m, int e) {
    if (m == 0) return 0.0;
    const int lz = clz64(m) - 11;               // to bit 52
    const int field = e - lz + 1075;
    if (field >= 1 && field <= 2046)
        return bits_double(((unsigned long long)field << 52) | ((m << lz) & 0xFFFFFFFFFFFFFull));
    return scalbn((double)m, e);
}

// The double-double of v 2^e, the top 106 bits of v.
__host__ __device__ __forceinline__ DD dd_of_int(__int128 v, int e) {
    const bool neg = v < 0;
    unsigned __int128 u = neg ? -(unsigned __int128)v : (unsigned __int128)v;
    if (u == 0) return DD{0.0, 0.0};
    const unsigned long long uh = (unsigned long long)(u >> 64);
    const int lz = uh ? clz64(uh) : 64 + clz64((unsigned long long)u);
    u <<= lz;                                   // leading bit at 127, weight of bit 0: 2^(e - lz)
    const double hi = scaled_int((unsigned long long)(u >> 75), e - lz + 75);
    const double lo = scaled_int((unsigned long long)(u >> 22) & ((1ull << 53) - 1), e - lz + 22);
    return neg ? DD{-hi, -lo} : DD{hi, lo};
}

// The double-double of v 2^(em - 1075 - top).  em is 0x7FF when a term was not
// finite: the sum is then NaN, as a double-double sum of such terms is.
__host__ __device__ __forceinline__ DD dd_of_fixed(__int128 v, int em, int top) {
    if (em >= 0x7FF) return DD{bits_double(0x7FF8000000000000ull), 0.0};
    return dd_of_int(v, em - 1075 - top);
}

__device__ __forceinline__ __int128 shfl_down128(__int128 v, int off) {
    const unsigned long long l = __shfl_down_sync(0xffffffffu, (unsigned long long)v, off);
    const unsigned long long h = __shfl_down_sync(0xffffffffu, (unsigned long long)((unsigned __int128)v >> 64), off);
    return (__int128)(((unsigned __int128)h << 64) | l);
}

__device__ __forceinline__ Partial zero_partial() {
    Partial p;
    p.sw = DD{0, 0};
    p.sw2 = DD{0, 0};
    p.npass = p.ntotal = p.ntries = p.nesc = 0;
    return p;
}

// Sum of the per-thread partials of a block: the largest exponents of all
// threads, the warps' sums as integers aligned to them, one thread adds those.
// Uses `scratch` (reduce_scratch_bytes(BLOCK) of shared memory, 16-byte
// aligned: the sums and, behind them, the exponents of the warps); result
// valid in thread 0.  All threads must call it.  (No shared memory of its own:
// the largest tiles leave 32 bytes of a block's.)
struct alignas(16) WarpSums {
    __int128 v[2];
    long long c[4];
};
static_assert(sizeof(WarpSums) == sizeof(Partial), "the scratch holds one per warp");

__host__ __device__ constexpr size_t reduce_scratch_bytes(int block) {
    return block / 32 * (sizeof(Partial) + 2 * sizeof(int));
}

template <int BLOCK>
__device__ __forceinline__ Partial block_reduce_partial(Partial a, Partial* scratch) {
    static_assert(BLOCK % 32 == 0 && BLOCK <= 1024, "whole warps");
    constexpr int NW = BLOCK / 32;
    constexpr int kTop = 61;   // 2 BLOCK <= 2048 terms of a sum below 2^(53 + kTop)
    WarpSums* sums = reinterpret_cast<WarpSums*>(scratch);
    int* s_em = reinterpret_cast<int*>(scratch + NW);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int em[2] = {(int)__reduce_max_sync(0xffffffffu, (unsigned)exponent_field(a.sw)),
                 (int)__reduce_max_sync(0xffffffffu, (unsigned)exponent_field(a.sw2))};
    if (lane == 0) {
        s_em[warp] = em[0];
        s_em[NW + warp] = em[1];
    }
    __syncthreads();
#pragma unroll
    for (int w = 0; w < NW; ++w) {
        em[0] = max(em[0], s_em[w]);
        em[1] = max(em[1], s_em[NW + w]);
    }
    WarpSums t{{fixed_of(a.sw, em[0], kTop), fixed_of(a.sw2, em[1], kTop)}, {a.npass, a.ntotal, a.ntries, a.nesc}};
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
#pragma unroll
        for (int q = 0; q < 2; ++q) t.v[q] += shfl_down128(t.v[q], off);
#pragma unroll
        for (int q = 0; q < 4; ++q) t.c[q] += __shfl_down_sync(0xffffffffu, t.c[q], off);
    }
    if (lane == 0) sums[warp] = t;
    __syncthreads();
    if (threadIdx.x == 0) {
#pragma unroll 1
        for (int w = 1; w < NW; ++w) {
            for (int q = 0; q < 2; ++q) t.v[q] += sums[w].v[q];
            for (int q = 0; q < 4; ++q) t.c[q] += sums[w].c[q];
        }
        a = Partial{dd_of_fixed(t.v[0], em[0], kTop), dd_of_fixed(t.v[1], em[1], kTop), t.c[0], t.c[1], t.c[2], t.c[3]};
    }
    return a;
}

}  // namespace heget
