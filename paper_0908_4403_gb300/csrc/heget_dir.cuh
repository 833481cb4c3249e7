// heget_dir.cuh -- the isotropic massless momenta of RAMBO (energy
// q0 = -ln(r2 r3), direction cos theta = 2 r0 - 1, phi = 2 pi r1; Sec. 2.1 eq.
// (4)) from random words, in integer arithmetic.
//
// GB300 issues a warp's FP64 instruction in 64 cycles of its sub-partition and
// a 32-bit integer or FP32 one in 1 - 2, so the FP64 form (two uniforms'
// conversions, a logarithm, a square root, a sine and cosine: about 50 FP64
// instructions a photon) was what bound the event generation.  Here every
// function works on 64-bit fixed-point numbers made of 32-bit multiplies, with
// more bits than FP64 carries: the uniforms enter exactly, cos theta is exact,
// sin theta, cos phi, sin phi and the energy's logarithm are within 2^-56 (the
// FP64 forms: 2^-53 to 2^-54), and each component of q is rounded to FP64
// once.  No sign is handled inside: angles are reduced to the first quadrant
// and logarithms to positive remainders.
//
// The functions run on the host too (their test compares them with
// high-precision values).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "heget_reduce.cuh"

#ifndef HEGET_DIR_TABLE
#define HEGET_DIR_TABLE static __device__ const
#endif
#include "heget_dirtab.h"

namespace heget {

typedef unsigned long long u64;
typedef unsigned int u32;

__host__ __device__ __forceinline__ u32 mulhi32(u32 a, u32 b) {
#ifdef __CUDA_ARCH__
    return __umulhi(a, b);
#else
    return (u32)(((u64)a * b) >> 32);
#endif
}

// (a b) >> 64 less at most 2 for a, b <= 2^63: three 32-bit multiply-adds (the
// product of the low words is left out).
__host__ __device__ __forceinline__ u64 mulhi63(u64 a, u64 b) {
    const u32 ah = (u32)(a >> 32), al = (u32)a, bh = (u32)(b >> 32), bl = (u32)b;
    const u64 t = (u64)ah * bl + (u64)al * bh;
    return (u64)ah * bh + (t >> 32);
}

// v 2^e rounded to double, v < 2^63, for results in the normal range; neg:
// with a minus sign.  The conversion is one instruction on the FP64 pipe; an
// integer one takes 40.  (v | 1 keeps zero out, half a unit of v's last place.)
__host__ __device__ __forceinline__ double double_of(u64 v, int e, bool neg) {
    const u64 b = double_bits((double)(long long)(v | 1u)) + ((u64)(long long)e << 52);
    return bits_double(neg ? b | (1ull << 63) : b);
}
// The same for normalised v (2^62 <= v < 2^63), by integer operations (ties away).
__host__ __device__ __forceinline__ double double_of_normal(u64 v, int e) {
    const u64 r = (v >> 10) + ((v >> 9) & 1u);             // 2^52 .. 2^53
    return bits_double(((u64)(e + 62 + 1022) << 52) + r);   // a carry of the rounding moves into the exponent
}

// The normalising left shift of a 128-bit product (h, l) and its top 64 bits
// after a shift by sh, 0 < sh < 128.  h = 0 happens once in 2^40 products: a
// branch of its own keeps its selects out of the common path.
__host__ __device__ __forceinline__ int clz_product(u64 h, u64 l) { return h ? clz64(h) : 64 + clz64(l); }
__host__ __device__ __forceinline__ u64 top_product(u64 h, u64 l, int sh) {
    if (sh >= 64) return l << (sh - 64);
    return (h << sh) | (l >> (64 - sh));
}

// The uniform u = (m + 1/2) 2^-52 of two random words (u01_from_words) as the
// odd integer 2 m + 1 = u 2^53.
__host__ __device__ __forceinline__ u64 u53_of_words(u32 lo, u32 hi) { return ((((u64)hi << 32) | lo) >> 11) | 1u; }

// A positive logarithm -ln(a b 2^-106) of odd a, b < 2^53 in units of 2^-72,
// as (hi, lo); error below 2^-62 absolute (2^-63 from the 64 bits kept of a
// b).  a b = M 2^(64 - lz), M in [2^63, 2^64): -ln = (lz - 22) ln 2 - ln m; with the table's
// R >= 1/m to 2^-9, t = m R - 1 in [0, 2^-9] is exact and
//   -ln m = ln R - ln(1 + t),
//   ln(1 + t) = t - t^2 (1/2 - t (1/3 - t (1/4 - t (1/5 - t/6))))   (next term 2^-65.8).
__host__ __device__ __forceinline__ unsigned __int128 neg_log(u64 a, u64 b, const uint4* logtab) {
    const unsigned __int128 P = (unsigned __int128)a * b;
    const u64 ph = (u64)(P >> 64), pl = (u64)P;
    const int lz = clz_product(ph, pl);
    const u64 M = top_product(ph, pl, lz);
#ifdef __CUDA_ARCH__
    const uint4 tb = __ldg(logtab + ((M >> 54) & 511u));
#else
    const uint4 tb = logtab[(M >> 54) & 511u];
#endif
    // D = M R - 2^94 = t 2^94; T = t 2^71
    const u64 d0 = (u64)(u32)M * tb.x;
    const u64 d1 = (u64)(u32)(M >> 32) * tb.x + (d0 >> 32) - (1ull << 62);
    const u64 T = (d1 << 9) | ((u32)d0 >> 23);
    const u32 th = (u32)(T >> 30);                                          // t 2^41
    const u32 k5 = 858993459u - mulhi32(th, 1398101u);                      // (1/5 - t/6) 2^32
    const u32 k4 = (1u << 30) - (mulhi32(th, k5) >> 9);                     // 1/4 - t (...)
    const u64 g = 3074457345618258603ull - ((u64)mulhi32(th, k4) << 22);    // (1/3 - t (...)) 2^63
    const u64 h = (1ull << 62) - (mulhi63(T, g) >> 7);                      // (1/2 - t (...)) 2^63
    const u64 l1 = (T << 1) - (mulhi63(mulhi63(T, T), h) >> 5);             // ln(1 + t) 2^72
    const u32 e = (u32)(lz - 22);
    const u64 p0 = (u64)e * kLn2W[0], p1 = (u64)e * kLn2W[1] + (p0 >> 32);
    const u32 p2 = e * kLn2W[2] + (u32)(p1 >> 32);
    unsigned __int128 V = ((unsigned __int128)p2 << 64) | (p1 << 32) | (u32)p0;
    V += ((unsigned __int128)tb.w << 64) | ((u64)tb.z << 32) | tb.y;
    return V - l1;
}

// cos and sin, in units of 2^-63, of the first-quadrant angle (pi/2) f 2^-51,
// f < 2^51 odd: table angle plus remainder th in [0, (pi/2)/512),
//   sin th = th - th^3 (1/6 - th^2/120),  cos th = 1 - (th^2/2 - th^4/24)
// (next terms 2^-59.6); within 2^-57.
__host__ __device__ __forceinline__ void quadrant_cos_sin(u64 f, const ulonglong2* angtab, u64& c, u64& s) {
    const u32 j = (u32)(f >> 42);
#ifdef __CUDA_ARCH__
    const ulonglong2 a = __ldg(angtab + j);
#else
    const ulonglong2 a = angtab[j];
#endif
    const u64 d = (f & ((1ull << 42) - 1)) << 21;             // remainder, 2^-63 of a table step
    const u64 th = mulhi63(d, kAngStep);                      // th 2^70
    const u64 t2 = mulhi63(th, th);                           // th^2 2^76
    const u32 t2n = (u32)(t2 >> 28);                          // th^2 2^48
    const u32 k3 = 2863311531u - mulhi32(t2n, 2184u);         // (1/6 - th^2/120) 2^34 (2^34/6, 2^18/120)
    const u32 w = mulhi32(t2n, k3);                           // th^2 (...) 2^50
    const u64 sn = th - (((u64)(u32)(th >> 30) * w) >> 20);   // sin th 2^70
    const u32 t4 = mulhi32(mulhi32(t2n, t2n), 0xAAAAAAABu);   // th^4 2/3 2^64 = th^4/24 2^68
    const u64 cm = (t2 >> 1) - ((u64)t4 << 8);                // (1 - cos th) 2^76
    // cos(a + th) = ca - (ca (1 - cos th) + sa sin th), sin(a + th) = sa + ca sin th - sa (1 - cos th)
    c = a.x - (((mulhi63(a.x, cm) >> 6) + mulhi63(a.y, sn)) >> 6);
    s = a.y + ((mulhi63(a.x, sn) - (mulhi63(a.y, cm) >> 6)) >> 6);
}

// An underestimate of 1/sqrt(x), x in [xh, xh + 1) 2^-32, by less than 2^-20 of it,
// in units of 2^-30 (FP32; rsqrtf is within 2 ulp; tested for every xh from 2^30).
__host__ __device__ __forceinline__ u32 root_estimate(u32 xh) {
#ifdef __CUDA_ARCH__
    const float y = rsqrtf(__uint2float_rn(xh) * 0x1p-32f);
    return __float2uint_rz(y * 1073741312.0f);         // y (1 - 2^-21) 2^30
#else
    const float y = 1.0f / __builtin_sqrtf((float)xh * 0x1p-32f);
    return (u32)(y * 1073741312.0f);
#endif
}

// sin theta in units of 2^-63 from a = 2^53 (1 + cos theta)/2 (odd):
// sin^2 theta = a (2^53 - a) 2^-104, exact in 106 bits, normalised by an even
// shift to x in [1/4, 1); with y an underestimate of 1/sqrt(x) (FP32, 2^-20)
// g = x y, d = (x - g^2) y / 2: sqrt(x) = g + d + (3/2) d^2 y + ... (the binomial series; next
// term 2^-59).
__host__ __device__ __forceinline__ u64 sin_theta(u64 a) {
    const unsigned __int128 P = (unsigned __int128)a * ((1ull << 53) - a);
    const u64 ph = (u64)(P >> 64), pl = (u64)P;
    const int ze = (clz_product(ph, pl) - 24) & ~1;
    const u64 X = top_product(ph, pl, 24 + ze);                // x 2^64
    const u32 xh = (u32)(X >> 32);
    const u32 Y = root_estimate(xh);
    const u64 g = ((u64)xh * Y << 1) + ((u64)(u32)X * Y >> 31);                 // x y 2^63
    const u64 e = (X >> 2) - mulhi63(g, g);                                     // (x - g^2) 2^62, below 2^43
    const u64 d = ((u64)(u32)(e >> 32) * Y << 1) + ((u64)(u32)e * Y >> 31);     // (x - g^2) y / 2 2^62
    const u32 dn = (u32)(d >> 12);                                              // 2^50
    const u32 d2 = mulhi32(mulhi32(dn, dn), Y);                                 // d^2 y 2^66
    return (g + (d << 1) + ((d2 + (d2 >> 1)) >> 3)) >> (ze >> 1);
}

// A positive V 2^-72, V < 2^80, as m 2^ex with 2^62 <= m < 2^63 (ex returned).
__host__ __device__ __forceinline__ int normal_of(unsigned __int128 V, u64& m) {
    const u64 h = (u64)(V >> 16);
    const u32 l = (u32)V & 0xFFFFu;
    const int lz = h ? clz64(h) : 64;
    m = lz < 64 ? ((h << lz) | (lz <= 16 ? (u64)((l << lz) >> 16) : (u64)l << (lz - 16))) >> 1
                : (u64)l << (clz64((u64)l) - 1);
    return lz < 64 ? 17 - lz - 72 : 1 - clz64((u64)l) - 72;
}

// q = q0 (1, sin th cos phi, sin th sin phi, cos th) of one photon from its
// four uniforms r0 .. r3 as odd integers (u53_of_words).
struct PhotonQ {
    double q0, q1, q2, q3;
};
__host__ __device__ __forceinline__ PhotonQ photon_q(u64 r0, u64 r1, u64 r2, u64 r3, const uint4* logtab,
                                                     const ulonglong2* angtab) {
    u64 m;
    const int ex = normal_of(neg_log(r2, r3, logtab), m);   // q0 = m 2^ex
    u64 c, s;
    quadrant_cos_sin(r1 & ((1ull << 51) - 1), angtab, c, s);
    const u32 quad = (u32)(r1 >> 51);
    const u64 ct = r0 >> 52 ? r0 - (1ull << 52) : (1ull << 52) - r0;     // |cos theta| 2^52
    const u64 st = sin_theta(r0);
    const u64 cp = quad & 1 ? s : c, sp = quad & 1 ? c : s;
    PhotonQ q;
    q.q0 = double_of_normal(m, ex);
    q.q1 = double_of(mulhi63(m, mulhi63(st, cp)), ex + 2, quad == 1 || quad == 2);
    q.q2 = double_of(mulhi63(m, mulhi63(st, sp)), ex + 2, quad >= 2);
    q.q3 = double_of(mulhi63(m, ct << 11), ex + 1, !(r0 >> 52));
    return q;
}

}  // namespace heget
