// heget_ps.cuh -- FP64 phase-space generation on the device: sqrt(s-hat)
// samplers, RAMBO flat massless n-body phase space (Sec. 2.1 eq. (4);
// Kleiss, Stirling, Ellis, CPC 40 (1986) 359), the photon cuts of Sec. 2.2
// eqs. (9)-(10), and the per-point record the amplitude kernels consume.
//
// GB300 executes FP64 at about 1/64 of the FP32 rate, so this file keeps
// FP64 for what needs it (RAMBO's boost; the Lorentz invariants behind the
// propagator denominators; cut decisions near a boundary): the isotropic
// momenta come from integer arithmetic of more bits (heget_dir.cuh), the cuts
// from FP32 where it decides, and square roots and reciprocals from FP32
// estimates refined in FP64.
#pragma once

#include "heget_common.cuh"
#include "heget_dir.cuh"
#include "heget_logtab.h"
#include "heget_sincostab.h"

namespace heget {

// Point record staged in shared memory between event generation (or input
// loading) and the amplitude rounds.  Momenta are divided by sqrt(s-hat) so
// that the FP32 chain works on O(1) numbers; the mass dimension 4 - 2n of
// |M|^2 is restored by `fac`.  The propagator denominators
//   t_T = (sum_{i in T} k_i - p2)^2 / s-hat,   T a proper photon subset,
// come from FP64: FP64 records and FP32 records up to n = 5 hold every t_T,
// computed in FP64 when the record is built (fill_denominators,
// set_denominator) and rounded once to R.  FP32 records from n = 6 hold the
// Lorentz invariants instead, t_T being a sum of them over T or, by momentum
// conservation (k_T - p2 = p1 - k_S, S = all - T), over its complement S,
//   t_T = sum_{i in T} d_i + sum_{i<j in T} s_ij = sum_{i in S} d'_i + sum_{i<j in S} s_ij,
//   d_i = k_i^2 - 2 k_i.p2,  d'_i = k_i^2 - 2 k_i.p1,  s_ij = 2 k_i.k_j,
// each computed in FP64 and kept as an unevaluated sum of two floats
// (hi + lo, about 48 significant bits); the rounds add up those of the
// smaller of T and S in float-float arithmetic (rec_denominator), so the
// FP32 chain again sees t_T with far more than FP32 accuracy, while the FP64
// pipe forms n(n+3)/2 invariants per point instead of 2^n - 2 sums.
template <class R, int N>
__host__ __device__ constexpr bool rec_invariants() {
    return sizeof(R) == sizeof(float) && N >= 6;
}
template <class R, int N, bool INV = rec_invariants<R, N>()>
struct RecDenominators {
    R t[1 << N];      // t_T by subset bitmask T (entries 0 and 2^n - 1 unused)
};
template <class R, int N>
struct RecDenominators<R, N, true> {
    float2 inv[N * (N + 3) / 2];   // (hi, lo): d_i at i, s_ij at N + pair_index(i, j), d'_i after them
};
template <class R, int N>
struct alignas(16) PointRec : RecDenominators<R, N> {
    double fac;       // (4 pi alpha Q^2)^n s-hat^(2-n): scaled sum -> |M|^2
    double wfac;      // scaled sum -> event weight (fb); 0 if masked
    R k[N][4];        // photon momenta / sqrt(s-hat)
    R e1, e2;         // energies of p1, p2 / sqrt(s-hat)  (p1 = e1 (1, 0, 0, 1), p2 = e2 (1, 0, 0, -1))
    R n1, n2;         // sqrt(2 e1), sqrt(2 e2): spinor normalisations
    R ssum;           // result of the tree: sum_h w_h |A_h|^2 in scaled units
    R kap2;           // sum_h w_h B_h^2, B_h >= sum over orderings |A_pi,h| (condition bound)
    int hsel;         // -1: every helicity; >= 0: only this lane (a sampled helicity); -2: none
    int valid;        // 0: amplitude not evaluated (bad input / sampler failure)
    int mask;         // passes the cuts
    int tries;        // outer sampler attempts
    int idx;          // the point's index within its tile or stage (records are compacted)
};

template <int N>
__host__ __device__ constexpr int pair_index(int i, int j) {  // i < j
    return i * N - i * (i + 1) / 2 + (j - i - 1);
}

// Flat massless n-body volume constant: Phi_n(s) = c_n s^(n-2) with
// c_n = (2 pi)^(4-3n) (pi/2)^(n-1) / ((n-1)! (n-2)!).
__host__ __device__ inline double phase_space_const(int n) {
    const double two_pi = 6.283185307179586476925287;
    const double half_pi = 1.570796326794896619231322;
    double f1 = 1, f2 = 1, c = 1;
    for (int i = 2; i <= n - 1; ++i) f1 *= i;
    for (int i = 2; i <= n - 2; ++i) f2 *= i;
    for (int i = 0; i < 3 * n - 4; ++i) c /= two_pi;
    for (int i = 0; i < n - 1; ++i) c *= half_pi;
    return c / (f1 * f2);
}

// FP32 estimate of the uniform u01_from_words(lo, hi) from its top 24 bits:
// |result - u| <= 2^-24.
__device__ __forceinline__ float u01_estimate(uint32_t hi) {
    return (__uint2float_rn(hi >> 8) + 0.5f) * 0x1p-24f;
}

// Toy-PDF momentum fraction: proposal x = u^2 (density ~ x^-1/2), accepted
// if v < (1-x)^3 (both uniforms from one Philox block per try); false when
// the bound of tries is hit.
//
// The acceptance test is the FP64 comparison v < (1 - u^2)^3, with the
// products and the difference rounded separately.  Most tries are settled
// first in FP32 from the same random bits: with |u_f - u|, |v_f - v| <= 2^-24,
// the FP32 value t_f of t = (1-u^2)^3 satisfies |t_f - t| <= 5.1 2^-24 (the
// input error through 3(1-u^2)^2 (2u + u^2 + 1/2) <= 3.1, plus two roundings
// of the cube), so |v_f - t_f| > 2^-20 = 16 2^-24 decides the comparison the
// same way; the FP64 test runs only inside that band (about 2e-6 of the
// tries).
//
// Integer and FP32 work (plus the rare FP64 tie-break) on the random words of
// one block.
__device__ __forceinline__ bool toy_pdf_accepts(const U4& w) {
    const float uf = u01_estimate(w.y), vf = u01_estimate(w.w);
    const float of = 1.0f - uf * uf;
    const float tf = of * of * of;
    if (vf < tf - 0x1p-20f) return true;
    if (vf > tf + 0x1p-20f) return false;
    const double u = u01_from_words(w.x, w.y), v = u01_from_words(w.z, w.w);
    const double om = __dsub_rn(1.0, __dmul_rn(u, u));
    return v < __dmul_rn(__dmul_rn(om, om), om);
}

// The accepted try's random words (false when the bound of tries is hit).
__device__ __forceinline__ bool toy_pdf_draw(const PointRng& rng, uint32_t& blk, int max_tries, uint32_t& wx,
                                             uint32_t& wy) {
    for (int t = 0; t < max_tries; ++t) {
        const U4 w = rng.words(kStreamSqrtS, blk++);
        if (toy_pdf_accepts(w)) {
            wx = w.x;
            wy = w.y;
            return true;
        }
    }
    return false;
}

__device__ __forceinline__ double toy_pdf_x_of(uint32_t wx, uint32_t wy) {
    const double u = u01_from_words(wx, wy);
    return __dmul_rn(u, u);
}

// Scalars of one generated event.  Its photon momenta in a MomView are those
// of RAMBO before the last scaling, with total (M, 0, 0, 0): times iM = 1/M
// they are in units of sqrt(s-hat) = rs, times rs iM in GeV.  ua, ub: the
// uniforms behind the toy PDF's fractions x = u^2, as integers u 2^53 (equal
// for the other samplers), so that e^y = sqrt(x1 / x2) = ua / ub.
struct EventInfo {
    double rs, iM;
    u64 ua, ub;
    int tries, ok, mask;
};

// The partonic frame's rapidity y = ln(x1 / x2) / 2 = ln ua - ln ub.
__device__ __forceinline__ double event_rapidity(const EventInfo& ev) {
    const __int128 d = (__int128)neg_log(ev.ub, 1ull << 53, kDirLog) - (__int128)neg_log(ev.ua, 1ull << 53, kDirLog);
    const bool neg = d < 0;
    const unsigned __int128 a = neg ? -(unsigned __int128)d : (unsigned __int128)d;   // y 2^72, below 2^80
    if (a == 0) return 0.0;
    u64 m;
    const int ex = normal_of(a, m);
    const double y = double_of_normal(m, ex);
    return neg ? -y : y;
}

// Helicity sampling (the paper's events carry one random helicity
// combination, Sec. 3): h = floor(2^(n+2) u) with u draw 0 of the helicity
// stream, bits as everywhere (bit 0 sigma1, bit 1 sigma2, bit 2 + i lambda_i).
// The kernels compute the lanes lambda with sigma1 = +, sigma2 = -; h with
// sigma1 = sigma2 vanishes exactly (-2: no lane), and h with sigma1 = -,
// sigma2 = + equals its parity image, the lane ~lambda.
template <int N>
__device__ __forceinline__ int sampled_lane(const PointRng& rng) {
    const U4 w = rng.words(kStreamHelicity, 0);
    const int h = (int)(u01_from_words(w.x, w.y) * (double)(1 << (N + 2)));
    const int s1 = h & 1, s2 = (h >> 1) & 1, lam = h >> 2;
    return s1 == s2 ? -2 : s1 ? lam : (~lam & ((1 << N) - 1));
}

// The record's lane selection (PointRec::hsel) for point i of stream seed:
// drawn when the record is written, so nothing stays live across RAMBO.
template <int N>
__device__ __forceinline__ int point_hsel(const Physics& ph, uint64_t seed, uint64_t i) {
    return ph.hel_sample ? sampled_lane<N>(PointRng(seed, i)) : -1;
}

// The sampler's random draws for one point, kept apart from the FP64 rest
// of the event: integer and FP32 work (plus a rare FP64 tie-break), which
// another set of threads can run ahead of time.  16 bytes: u01_from_words
// ignores the low 12 bits of its low word, so those of ax carry the outer
// attempts and the success flag.
struct alignas(16) SampleDraw {
    uint32_t ax, ay;   // toy PDF: words of the accepted x1 draw; uniform: the words of sqrt(s-hat)
    uint32_t bx, by;   // toy PDF: words of the accepted x2 draw
    __device__ __forceinline__ int tries() const { return (int)((ax >> 1) & 0x7FFu); }
    __device__ __forceinline__ int ok() const { return (int)(ax & 1u); }
    __device__ __forceinline__ void set(int tries, int ok) { ax = (ax & ~0xFFFu) | ((uint32_t)tries << 1) | (uint32_t)ok; }
};

// The floor test r > floor, r = 2 E sqrt(x1 x2) in FP64, of a draw's two
// fractions: the test u_a u_b > floor / (2 E) on the uniforms behind x = u^2,
// whose FP32 estimates (within 2^-24) settle it outside a band of +-16 2^-24
// around the threshold; the FP64 r decides inside it.
__device__ __forceinline__ bool above_floor(const SamplerArgs& S, const SampleDraw& d) {
    const float p = u01_estimate(d.ay) * u01_estimate(d.by);
    if (p > S.band_hi) return true;
    if (p < S.band_lo) return false;
    const double a = toy_pdf_x_of(d.ax, d.ay), b = toy_pdf_x_of(d.bx, d.by);   // rare
    return 2.0 * S.e_beam * sqrt(a * b) > S.floor;
}

__device__ __forceinline__ SampleDraw sample_draw(const SamplerArgs& S, const PointRng& rng) {
    SampleDraw d{0u, 0u, 0u, 0u};
    if (S.kind == HEGET_SAMPLER_FIXED) {
        d.set(1, 1);
        return d;
    }
    if (S.kind == HEGET_SAMPLER_UNIFORM) {
        const U4 w = rng.words(kStreamSqrtS, 0);
        d.ax = w.x;
        d.ay = w.y;
        d.set(1, 1);
        return d;
    }
    uint32_t blk = 0;
    int tries = S.max_tries, ok = 0;
    for (int t = 1; t <= S.max_tries; ++t) {
        if (!toy_pdf_draw(rng, blk, S.max_tries, d.ax, d.ay)) break;
        if (!toy_pdf_draw(rng, blk, S.max_tries, d.bx, d.by)) break;
        if (above_floor(S, d)) {
            tries = t;
            ok = 1;
            break;
        }
    }
    d.set(tries, ok);
    return d;
}

// The draws (sample_draw) of the cnt events index(0 .. cnt - 1) of a stream
// into out, by one warp.  The toy PDF's rejection loops take five blocks of
// random words an event on average and fifteen in the slowest of 32, so a lane
// that has finished an event takes the next one, and every pass of the loop
// tests one block in (nearly) every lane: about 28 passes for 128 events
// instead of 4 x 15, 20 instructions an event instead of 53.  All lanes must
// call it; the caller synchronises before other warps read out.
template <class Index>
__device__ __forceinline__ void warp_draws(const SamplerArgs& S, uint64_t seed, const Index& index, int cnt,
                                           SampleDraw* out) {
    const int lane = threadIdx.x & 31;
    if (S.kind != HEGET_SAMPLER_TOY_PDF) {
        for (int p = lane; p < cnt; p += 32) out[p] = sample_draw(S, PointRng(seed, index(p)));
        return;
    }
    int e = lane, next = 32;
    bool active = e < cnt, second = false;
    uint32_t blk = 0;
    int t = 1, inner = 0;
    SampleDraw d{0u, 0u, 0u, 0u};
    while (__any_sync(0xffffffffu, active)) {
        bool done = false;
        if (active) {
            const U4 w = PointRng(seed, index(e)).words(kStreamSqrtS, blk++);
            int ok = 0;
            if (toy_pdf_accepts(w)) {
                inner = 0;
                if (!second) {
                    d.ax = w.x;
                    d.ay = w.y;
                } else {
                    d.bx = w.x;
                    d.by = w.y;
                    ok = above_floor(S, d);
                    done = ok || t == S.max_tries;
                    t += !ok;
                }
                second = !second;
            } else {
                done = ++inner == S.max_tries;
            }
            if (done) {
                d.set(ok ? t : S.max_tries, ok);
                out[e] = d;
            }
        }
        const unsigned fin = __ballot_sync(0xffffffffu, done);
        if (done) {
            e = next + __popc(fin & ((1u << lane) - 1u));
            active = e < cnt;
            second = false;
            blk = 0;
            t = 1;
            inner = 0;
        }
        next += __popc(fin);
    }
}

// sqrt(s-hat) and the outer attempts from the draws: 2 E sqrt(x1 x2) = 2 E ua
// ub, with the product of the uniforms rounded once.
__device__ __forceinline__ void sample_finish(const SamplerArgs& S, const SampleDraw& d, EventInfo& ev) {
    ev.ok = d.ok();
    ev.tries = d.tries();
    ev.ua = ev.ub = 1ull << 52;   // e^y = 1, in the middle of FP32's range
    if (S.kind == HEGET_SAMPLER_FIXED) {
        ev.rs = S.sqrt_s;
    } else if (S.kind == HEGET_SAMPLER_UNIFORM) {
        ev.rs = S.lo + (S.hi - S.lo) * u01_from_words(d.ax, d.ay);
    } else if (ev.ok) {
        ev.ua = u53_of_words(d.ax, d.ay);
        ev.ub = u53_of_words(d.bx, d.by);
        const unsigned __int128 P = (unsigned __int128)ev.ua * ev.ub;
        const int lz = clz_product((u64)(P >> 64), (u64)P);
        ev.rs = 2.0 * S.e_beam * double_of_normal(top_product((u64)(P >> 64), (u64)P, lz) >> 1, 65 - lz - 106);
    } else {
        ev.rs = S.floor;
    }
}

// Photon momenta of one point held in shared memory: slot (a, m) at
// p[(slots a + m) * stride], m = 0..3 the components (E, px, py, pz).
// Generated points use slots = kMomSlots with stride = points of the tile
// (point-minor layout: consecutive threads touch consecutive words); input
// rows use slots = 4, stride = 1.
constexpr int kMomSlots = 4;

struct MomView {
    double* p;
    int stride;
    int slots;
    __device__ __forceinline__ double& operator()(int a, int m) const { return p[(slots * a + m) * stride]; }
};

// double -> float, rounded to nearest even, by integer operations on the bit
// pattern: on GB300 the hardware conversion occupies the FP64 pipe, which
// the event generation saturates.  Exact for results in the normal float
// range; results below it become a signed zero (no subnormals), above it
// +-inf, and NaN stays NaN.
__device__ __forceinline__ float f32_rn(double x) {
    // 32-bit words throughout: the round bit is bit 28 of lo, the sticky bits
    // 0..27, the kept bits start at 29; the exponent field of
    // (|x| >> 29) mod 2^32 minus (1023 - 127) << 23 is the float's, and a
    // round-up carry out of the mantissa moves into it
    const unsigned int hi = (unsigned int)__double2hiint(x), lo = (unsigned int)__double2loint(x);
    const unsigned int habs = hi & 0x7FFFFFFFu, sign = hi & 0x80000000u;
    const unsigned int t = __funnelshift_r(lo, habs, 29);          // exponent and top mantissa bits
    const unsigned int inc = (lo >> 28) & ((lo & 0x2FFFFFFFu) != 0u ? 1u : 0u);   // round bit and (sticky or lsb)
    unsigned int f = t - (896u << 23) + inc;
    f = habs < 0x38100000u ? 0u : f;
    f = habs >= 0x47F00000u ? ((habs > 0x7FF00000u || (habs == 0x7FF00000u && lo != 0u)) ? 0x7FC00000u : 0x7F800000u) : f;
    return __uint_as_float(f | sign);
}

// A record field from its FP64 value: f32_rn for FP32 records.
template <class R>
__device__ __forceinline__ R rec_value(double x) {
    if constexpr (sizeof(R) == sizeof(float)) return f32_rn(x);
    else return x;
}

// Natural logarithm of a positive normal double by Tang's table-driven method
// (P. T. P. Tang, ACM TOMS 16 (1990) 378): x = 2^e m with m in [1, 2), F the
// nearest breakpoint 1 + j/256, f = m - F (exact, |f| <= 1/512), r = f / F,
//   ln x = e ln 2 + ln F + ln(1 + r),
// with ln F and ln 2 from double-double tables (heget_logtab.h) and ln(1 + r)
// by its series to r^6 (|r| <= 2^-9: truncation below 2^-56 relative).  F and
// e become doubles through their bit patterns, so the whole costs 15 FP64
// operations instead of a general-purpose logarithm.  (An entry point of its
// own, heget_log_table; the generator's energies come from neg_log.)
__device__ __forceinline__ double log_table(double x) {
    const int hi = __double2hiint(x), lo = __double2loint(x);
    const int e = ((hi >> 20) & 0x7FF) - 1023;
    const double m = __hiloint2double((hi & 0x000FFFFF) | 0x3FF00000, lo);
    const int j = (((hi >> 11) & 0x1FF) + 1) >> 1;            // nearest breakpoint, 0 .. 256
    const double F = __hiloint2double(0x3FF00000 + (j << 12), 0);   // 1 + j/256
    const double f = m - F;                                          // exact
    const double r = f * __ldg(&kLogTab[j][2]);
    // ln(1 + r) - r = r^2 (-1/2 + r (1/3 + r (-1/4 + r (1/5 - r/6))))
    double q = -1.0 / 6.0;
    q = fma(q, r, 0.2);
    q = fma(q, r, -0.25);
    q = fma(q, r, 1.0 / 3.0);
    q = fma(q, r, -0.5);
    const double p = r * r * q;
    // e as a double: 2^52 + 2^31 + e carries e in its low mantissa bits
    const double ed = __hiloint2double(0x43300000, (int)(0x80000000u + (unsigned)e)) - 0x1.00000800p52;
    const double lhi = fma(ed, kLn2Hi, __ldg(&kLogTab[j][0]));
    const double llo = fma(ed, kLn2Lo, __ldg(&kLogTab[j][1]));
    return lhi + (r + (p + llo));
}

// cos and sin of the RAMBO azimuth phi = 2 pi r for the uniform
// r = u01_from_words(lo, hi) = (2m + 1) 2^-53, m the top 52 bits of (hi, lo),
// by a breakpoint table (heget_sincostab.h): j = round(512 r), a = 2 pi j/512
// and theta = 2 pi (r - j/512), |theta| <= pi/512.  The remainder is exact:
// r - j/512 = D 2^-53 with the integer D = 2m + 1 - j 2^44, |D| <= 2^43.  With
// s = sin theta and c' = cos theta - 1 by their Taylor series (truncated below
// 1e-19),
//   cos phi = cos a + (c' cos a - s sin a),  sin phi = sin a + (c' sin a + s cos a),
// within about 2 ulp; 15 FP64 operations and one table load.  (An entry point of
// its own, heget_sincos_2pi; the generator's azimuth is quadrant_cos_sin.)
__device__ __forceinline__ void sincos_2pi_words(uint32_t lo, uint32_t hi, double& sp, double& cp) {
    const unsigned long long m = ((((unsigned long long)hi) << 32) | lo) >> 12;
    const unsigned long long j = (m + (1ull << 42)) >> 43;   // 0 .. 512
    const long long D = (long long)(2 * m + 1) - (long long)(j << 44);
    // D as a double without a conversion: 1.5 2^52 + D has D in its mantissa
    const double d = __longlong_as_double(0x4338000000000000ll + D) - 0x1.8p52;
    const double th = d * 0x1.921fb54442d18p-51;   // 2 pi 2^-53
    const double t2 = th * th;
    const double s = fma(th * t2, fma(t2, 1.0 / 120.0, -1.0 / 6.0), th);
    const double cm = t2 * fma(t2, fma(t2, -1.0 / 720.0, 1.0 / 24.0), -0.5);
    const double2 a = __ldg(&kSinCosTab[j & (kSinCosTable - 1)]);
    cp = a.x + fma(a.x, cm, -(a.y * s));
    sp = a.y + fma(a.y, cm, a.x * s);
}

// Inverse square root and reciprocal of a double in the normal float range
// (with a margin): an FP32 estimate (relative error e/2 or e about 2^-22) and
// one step of the binomial series to e^2 in FP64,
//   x^-1/2 = y (1 + e/2 + 3/8 e^2 + ...), e = 1 - x y^2;  1/x = y (1 + e + e^2 + ...), e = 1 - x y
// (next terms below 2^-63): 5 and 3 FP64 operations.
__device__ __forceinline__ double f64_of_f32(float f);
__device__ __forceinline__ double rsqrt_series(double x) {
    const double y = f64_of_f32(rsqrtf(f32_rn(x)));
    const double e = fma(-x * y, y, 1.0);
    return fma(y * e, fma(0.375, e, 0.5), y);
}
__device__ __forceinline__ double recip_series(double x) {
    const double y = f64_of_f32(__frcp_rn(f32_rn(x)));
    const double e = fma(-x, y, 1.0);
    return fma(y, fma(e, e, e), y);
}

// RAMBO: n massless momenta with total (M, 0, 0, 0), and iM = 1/M.  Photon i
// uses draws 4i..4i+3 of the RAMBO stream: cos(theta) = 2 r0 - 1, phi = 2 pi
// r1, q0 = -ln(r2 r3) (photon_q); the isotropic q_i are boosted to the rest
// frame of their sum.
//
// GB300, FP64 instructions a point, before -> after: 403 -> 154 at n = 4, 500,000
// phase-space points at n = 5 454 -> 226 us (230 now, with the guards for parallel
// photons; unrolling the loops by 2 or 4: no gain, more instruction-cache
// misses).  True error of the momenta (against
// quad precision, 2-norm): n = 5 2.71e-16 -> 2.69e-16, n = 2 3.2e-14 -> 2.4e-14.
template <int N>
__device__ __forceinline__ double rambo(const PointRng& rng, const MomView& v) {
    double Q0 = 0, Q1 = 0, Q2 = 0, Q3 = 0;
#pragma unroll 1
    for (int i = 0; i < N; ++i) {
        const U4 w = rng.words(kStreamRambo, 2 * i), z = rng.words(kStreamRambo, 2 * i + 1);
        const PhotonQ q = photon_q(u53_of_words(w.x, w.y), u53_of_words(w.z, w.w), u53_of_words(z.x, z.y),
                                   u53_of_words(z.z, z.w), kDirLog, kDirAng);
        v(i, 0) = q.q0;
        v(i, 1) = q.q1;
        v(i, 2) = q.q2;
        v(i, 3) = q.q3;
        Q0 += q.q0;
        Q1 += q.q1;
        Q2 += q.q2;
        Q3 += q.q3;
    }
    // M = sqrt(Q^2), b = -Q/M, gamma = Q0/M, a = 1/(1 + gamma) = M/(M + Q0):
    // p_i = (gamma q0 + b.q, q + b (q0 + a b.q)).
    const double M2 = Q0 * Q0 - Q1 * Q1 - Q2 * Q2 - Q3 * Q3;
    // (all photons parallel to rounding: the library's root, NaN below 0)
    const double iM = __double2hiint(M2) > 0x39B00000 ? rsqrt_series(M2) : rsqrt(M2);   // M2 > 8e-31
    const double M = M2 * iM;
    const double b1 = -Q1 * iM, b2 = -Q2 * iM, b3 = -Q3 * iM;
    const double a = M * recip_series(M + Q0);
    const double g = Q0 * iM;
#pragma unroll 1
    for (int i = 0; i < N; ++i) {
        const double q0 = v(i, 0), q1 = v(i, 1), q2 = v(i, 2), q3 = v(i, 3);
        const double bq = b1 * q1 + b2 * q2 + b3 * q3;
        const double t = fma(a, bq, q0);
        v(i, 0) = fma(g, q0, bq);
        v(i, 1) = fma(b1, t, q1);
        v(i, 2) = fma(b2, t, q2);
        v(i, 3) = fma(b3, t, q3);
    }
    return iM;
}

// a < b for doubles a, b >= +0 (squares and their products, never -0 or
// NaN): their IEEE bit patterns order like the values, so the comparison
// runs on the integer pipe, not on the FP64 pipe with the arithmetic.
__device__ __forceinline__ bool lt_nonneg(double a, double b) {
    return __double_as_longlong(a) < __double_as_longlong(b);
}

// v < 0 from the bit pattern (false for -0).
__device__ __forceinline__ bool is_negative(double v) {
    const long long b = __double_as_longlong(v);
    return b < 0 && (b << 1) != 0;
}

// v < a * w, decided on squares (w >= 0): no square root; written with
// selects, so the lanes of a warp stay together.
__device__ __forceinline__ bool lt_scaled(double v, double a, double w2) {
    const double v2 = v * v, r2 = a * a * w2;
    const bool neg = is_negative(v);
    return a >= 0 ? (neg || lt_nonneg(v2, r2)) : (neg && lt_nonneg(r2, v2));
}

// Photon cuts, strict (Sec. 2.2): pT > pt_min, |eta + y| < eta_max with
// eta = asinh(pz / pT), and Delta R = sqrt(Delta eta^2 + Delta phi^2) > dr_min
// for every pair (Delta phi in [0, pi]); dr_min <= 0 disables Delta R.
// Evaluated without per-photon transcendentals:
//   eta + y in (-E, E)  <=>  pz / pT in (sinh(-E - y), sinh(E - y)),
//     sinh(E -+ y) = sinh E cosh y -+ cosh E sinh y with e^y = sqrt(x1/x2);
//   sinh(eta_i - eta_j) = (pz_i E_j - pz_j E_i) / (pT_i pT_j)   (|p| = E),
//   cos(phi_i - phi_j)  = (px_i px_j + py_i py_j) / (pT_i pT_j);
// a pair passes at once if |Delta eta| > R or Delta phi > R (compared on
// squares), and only the remaining close pairs evaluate asinh and atan2.
// The momenta are in units of 1/scale GeV (EventInfo).  Out of line: only
// points that the FP32 tests leave open come here.
template <int N>
__device__ __noinline__ int pass_cuts(const MomView p, double scale, u64 ua, u64 ub, const Physics& ph) {
    // every photon and pair is tested without early exits: the FP64 pipe
    // executes whole warps, so a lane that could stop early saves nothing and
    // the divergence would cost the others
    const double ey = (double)ua / (double)ub, iey = (double)ub / (double)ua;   // e^y, e^-y
    const double shy = 0.5 * (ey - iey), chy = 0.5 * (ey + iey);
    const double s_hi = ph.sinh_eta * chy - ph.cosh_eta * shy;    // sinh(E - y)
    const double s_lo = -ph.sinh_eta * chy - ph.cosh_eta * shy;   // sinh(-E - y)
    const double pt_min = ph.pt_min / scale, pt2min = pt_min * pt_min;
    bool ok = p(0, 0) == p(0, 0);   // (the comparisons on bits below do not know NaN)
    double pt2[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const double pz = p(i, 3);
        pt2[i] = p(i, 1) * p(i, 1) + p(i, 2) * p(i, 2);
        // pT > pt_min and s_lo pT < pz < s_hi pT
        ok = ok & lt_nonneg(pt2min, pt2[i]) & lt_scaled(pz, s_hi, pt2[i]) & lt_scaled(-pz, -s_lo, pt2[i]);
    }
    if (ph.dr_min > 0) {
        // squares only: |p| = E for massless photons, and the sinh / cos
        // comparisons are decided on squares; pT_i pT_j (a square root) is
        // formed only for the close pairs that need asinh and atan2.  The
        // pairs are screened first (pair_index bits of `close`), then the
        // close ones, which are rare, settled one by one.
        const double sdr2 = ph.sinh_dr * ph.sinh_dr;
        unsigned close = 0;
#pragma unroll
        for (int i = 0; i < N; ++i)
#pragma unroll
            for (int j = i + 1; j < N; ++j) {
                const double pp2 = pt2[i] * pt2[j];                      // (pT_i pT_j)^2
                const double sh = p(i, 3) * p(j, 0) - p(j, 3) * p(i, 0);   // sinh(d eta) pT_i pT_j
                const double dot = p(i, 1) * p(j, 1) + p(i, 2) * p(j, 2);  // cos(d phi) pT_i pT_j
                const bool far = lt_nonneg(sdr2 * pp2, sh * sh) | lt_scaled(dot, ph.cos_dr, pp2);
                close |= (far ? 0u : 1u) << pair_index<N>(i, j);
            }
        if (!ok) close = 0;
        while (close) {
            int q = __ffs(close) - 1, i = 0;
            close &= close - 1;
            while (q >= N - 1 - i) q -= N - 1 - i++;
            const int j = i + 1 + q;
            const double xi = p(i, 1), yi = p(i, 2), zi = p(i, 3);
            const double xj = p(j, 1), yj = p(j, 2), zj = p(j, 3);
            const double pp2 = (xi * xi + yi * yi) * (xj * xj + yj * yj);
            const double sh = zi * p(j, 0) - zj * p(i, 0);
            const double dot = xi * xj + yi * yj;
            // a close pair: |d eta|, d phi <= R.  With s = |sinh d eta| and
            // t = tan d phi (dot > 0 here when R < pi/2),
            //   s^2 (1 - s^2/6)^2 <= d eta^2 <= s^2,
            //   t^2 (1 - t^2/3)^2 <= d phi^2 <= t^2
            // (asinh and atan lie between their first two Taylor terms and
            // their first), which settles all but the pairs within about 1 %
            // of R; those take asinh and atan2.
            const double cr = xi * yj - yi * xj;
            const double R2 = ph.dr_min * ph.dr_min;
            bool exact = !(dot > 0);
            if (!exact) {
                const double s2 = sh * sh / pp2, t2 = cr * cr / (dot * dot);
                const double a = 1.0 - s2 * (1.0 / 6.0), b = 1.0 - t2 * (1.0 / 3.0);
                const double hi = s2 + t2, lo = s2 * a * a + t2 * b * b;
                if (!(a > 0 && b > 0)) {
                    exact = true;   // wide cuts (R beyond about 1): the lower bounds do not hold
                } else if (lo > R2 * (1.0 + 1e-12)) {
                    // Delta R > R: the pair passes
                } else if (hi < R2 * (1.0 - 1e-12)) {
                    ok = false;
                } else {
                    exact = true;
                }
            }
            if (exact) {   // rare
                const double ptt = sqrt(pp2);
                const double deta = asinh(sh / ptt);
                const double dphi = atan2(fabs(cr), dot);
                ok = ok && deta * deta + dphi * dphi > R2;
            }
            if (!ok) close = 0;
        }
    }
    return ok ? 1 : 0;
}

// x as a float for the FP32 cut decisions: truncated towards zero (relative
// error below 2^-23; zero below the normal float range) by three integer
// operations on the bits.  x must be a number below the float range's end
// (anything else becomes some number: fp32_holds comes first).
__device__ __forceinline__ float f32_cut(double x) {
    const unsigned int hi = (unsigned int)__double2hiint(x), lo = (unsigned int)__double2loint(x);
    const unsigned int f = __funnelshift_l(lo, hi, 3) - (384u << 23);   // 9 exponent bits rebased by 896 mod 512
    const bool tiny = (hi & 0x7FFFFFFFu) < 0x38100000u;
    return tiny ? 0.0f : __uint_as_float((f & 0x7FFFFFFFu) | (hi & 0x80000000u));
}

// Whether FP32 holds an event's scale.  Not where the photons are parallel to
// rounding: their mass M is then tiny or not a number, and so may be the
// momenta, which f32_cut would turn into numbers.
__device__ __forceinline__ bool fp32_holds(const EventInfo& ev) {
    // rs in (0.01, 1e8), 1/M below 1e12, on the high words: larger for infinities, NaN and negative values
    const unsigned r = (unsigned)__double2hiint(ev.rs), m = (unsigned)__double2hiint(ev.iM);
    return r > 0x3F847AE1u && r < 0x4197D784u && m < 0x426D1A94u;
}

// The cut decisions in FP32 wherever FP32 settles them: the same decisions as
// pass_cuts, which decides the points that stay open.  With u = 2^-24, the
// truncated components carry 2 u.  Rapidities enter through the light-cone
// components p+ = E + pz, p- = pT^2 / p+ (for pz >= 0; the other way round
// below 0), which do not cancel:
//   eta + y < E  <=>  p+ e^y < e^2E p- e^-y,
//   sinh(eta_i - eta_j) pT_i pT_j = (p+_i p-_j - p-_i p+_j) / 2,
// all terms within about 20 u, so 64 u of relative margin (32 u of the terms'
// magnitudes for the two sides of the difference, 16 u for cos(d phi) pT pT)
// is safe.  A pair that is not surely far in eta or phi takes asinhf and
// atan2f (3 ulp each): d eta and d phi within 32 u absolute, and Delta R^2
// open only within 2 (d eta + d phi) 32 u of R^2.  About 3e-4 of the points
// stay open (n = 4, toy PDF).
//
// Bound: the FP64 tests cost 24 + 10 n (n - 1) / 2 FP64 instructions a point
// (90 of 545 at n = 4) at 64 cycles each per warp; these cost about 70 n + 20
// n (n - 1) / 2 FP32 and integer instructions at 1 - 2 cycles.  GB300, before ->
// after: n = 4 step of 1,048,576 points 1123 -> 1012 us, phase space of 500,000
// points at n = 5 668 -> 454 us (this form alone; both are faster by now: rambo).
//
// The momenta are in RAMBO's units (total M, of the order of n), which FP32
// holds; pT is compared in GeV.  Energies, pT cuts, boosts (u below 2^-30), e^2E
// and sinh^2 R that FP32 does not hold are left to pass_cuts, and so is a photon whose pT^2 FP32
// cannot hold accurately.
template <int N>
__device__ __forceinline__ int pass_cuts_fast(const MomView& p, const EventInfo& ev, const Physics& ph) {
    constexpr float kU = 5.9604645e-8f;   // 2^-24
    const double scale = ev.rs * ev.iM;
    if (!(fp32_holds(ev) && ph.eta_max < 40.0 && ph.dr_min < 20.0 && ph.pt_min < 1e12 &&
          !(ph.pt_min > 0 && ph.pt_min < 1e-12) &&
          ev.ua >> 23 != 0 && ev.ub >> 23 != 0))
        return pass_cuts<N>(p, scale, ev.ua, ev.ub, ph);
    constexpr float kLo = 1.0f - 64.0f * kU, kHi = 1.0f + 64.0f * kU;
    // e^y = ua / ub: a and b below are p+ e^y and p- e^-y times ua ub 2^-106
    const float uaf = __ull2float_rz(ev.ua) * 0x1p-53f, ubf = __ull2float_rz(ev.ub) * 0x1p-53f;
    const float eyf = uaf * uaf, ieyf = ubf * ubf, s2 = f32_cut(scale) * f32_cut(scale);
    const float eE = f32_cut(ph.sinh_eta) + f32_cut(ph.cosh_eta), e2E = eE * eE;
    const float ptmin2 = f32_cut(ph.pt_min) * f32_cut(ph.pt_min);
    float x[N], y[N], pp[N], pm[N], pt2[N];
    bool fail = false, open = false;   // some test surely fails; some test is not decided
#pragma unroll
    for (int i = 0; i < N; ++i) {
        const float e = f32_cut(p(i, 0)), z = f32_cut(p(i, 3));
        x[i] = f32_cut(p(i, 1));
        y[i] = f32_cut(p(i, 2));
        pt2[i] = x[i] * x[i] + y[i] * y[i];
        const float big = e + fabsf(z), small = __fdividef(pt2[i], big);
        pp[i] = z < 0.0f ? small : big;
        pm[i] = z < 0.0f ? big : small;
        const bool held = pt2[i] > 1e-30f;
        const float pt2g = pt2[i] * s2;   // GeV^2
        fail = fail || pt2g < ptmin2 * kLo;
        open = open || !(held && pt2g > ptmin2 * kHi);
        const float a = pp[i] * eyf, b = pm[i] * ieyf;
        fail = fail || (held && (a * kLo > e2E * b || b * kLo > e2E * a));
        open = open || !(a * kHi < e2E * b && b * kHi < e2E * a);
    }
    unsigned close = 0;
    if (ph.dr_min > 0) {
        const float sdr = f32_cut(ph.sinh_dr), sdr2 = sdr * sdr, cdr = f32_cut(ph.cos_dr);
#pragma unroll
        for (int i = 0; i < N; ++i)
#pragma unroll
            for (int j = i + 1; j < N; ++j) {
                const float pp2 = pt2[i] * pt2[j];
                const float u = pp[i] * pm[j], v = pm[i] * pp[j];
                const float sh = fabsf(u - v) - 32.0f * kU * (u + v);   // twice |sinh(d eta)| pT pT, from below
                const float xx = x[i] * x[j], yy = y[i] * y[j];
                const float dot = xx + yy + 16.0f * kU * (fabsf(xx) + fabsf(yy));   // from above
                const float c = cdr * (pp2 * rsqrtf(pp2));
                const bool far = (sh > 0.0f && sh * sh * 0.25f > sdr2 * pp2 * kHi) || dot < c - 64.0f * kU * fabsf(c);
                close |= (far ? 0u : 1u) << pair_index<N>(i, j);
            }
    }
    if (fail) return 0;
    const float R = f32_cut(ph.dr_min), R2 = R * R;
    while (close) {
        int q = __ffs(close) - 1, i = 0;
        close &= close - 1;
        while (q >= N - 1 - i) q -= N - 1 - i++;
        const int j = i + 1 + q;
        const float xi = f32_cut(p(i, 1)), yi = f32_cut(p(i, 2)), zi = f32_cut(p(i, 3));
        const float xj = f32_cut(p(j, 1)), yj = f32_cut(p(j, 2)), zj = f32_cut(p(j, 3));
        const float ti = xi * xi + yi * yi, tj = xj * xj + yj * yj;
        const float bi = f32_cut(p(i, 0)) + fabsf(zi), bj = f32_cut(p(j, 0)) + fabsf(zj);
        const float si = __fdividef(ti, bi), sj = __fdividef(tj, bj);
        const float u = (zi < 0.0f ? si : bi) * (zj < 0.0f ? bj : sj), v = (zi < 0.0f ? bi : si) * (zj < 0.0f ? sj : bj);
        const float deta = asinhf(0.5f * fabsf(u - v) * rsqrtf(ti * tj));
        const float dphi = atan2f(fabsf(xi * yj - yi * xj), xi * xj + yi * yj);
        const float d2 = deta * deta + dphi * dphi;
        const float m = 64.0f * kU * (deta + dphi + 64.0f * kU) + 8.0f * kU * R2;
        if (d2 < R2 - m) return 0;
        open = open || !(d2 > R2 + m);
    }
    return open ? pass_cuts<N>(p, scale, ev.ua, ev.ub, ph) : 1;
}

// Event i of stream `seed` from its sampler draws d: sqrt(s-hat), RAMBO
// momenta into v (units of EventInfo), cut decision.
template <int N>
__device__ __forceinline__ void generate_from(const PointRng& rng, const SampleDraw& d, const SamplerArgs& S,
                                              const Physics& ph, const MomView& v, EventInfo& ev) {
    sample_finish(S, d, ev);
    ev.iM = rambo<N>(rng, v);
    ev.mask = ev.ok ? pass_cuts_fast<N>(v, ev, ph) : 0;
}

template <int N>
__device__ __forceinline__ void generate_event(uint64_t seed, uint64_t i, const SamplerArgs& S, const Physics& ph,
                                               const MomView& v, EventInfo& ev) {
    const PointRng rng(seed, i);
    generate_from<N>(rng, sample_draw(S, rng), S, ph, v, ev);
}

// Flat phase-space weight Phi_n(s) of eq. (4).
template <int N>
__device__ __forceinline__ double phase_space_weight(double s) {
    double sn2 = 1;
    for (int a = 2; a < N; ++a) sn2 *= s;
    return phase_space_const(N) * sn2;
}

// Propagator denominators t_T of the record, in FP64, from photon momenta p
// and p2 = E2 (1, 0, 0, -1), times `is` if SCALE (momenta in GeV, is =
// 1/s-hat; without SCALE the momenta are already divided by sqrt(s-hat)).
// For n <= 5 they are sums of the Lorentz invariants
//   t_T = sum_{i in T} d_i + sum_{i<j in T} s_ij,
//   d_i = k_i^2 - 2 k_i.p2,  s_ij = 2 k_i.k_j,
// built up over the sets in increasing order in registers: with h the
// highest photon of T and U = T - {h},
//   t_T = t_U + e_h(U),  e_h(U) = d_h + sum_{j in U} s_jh = e_h(U - {l}) + s_lh
// (l the lowest photon of U): two additions per set.  Larger n: FP64
// records use set_denominator, FP32 records keep the invariants
// (rec_invariant).
template <class R, int N, bool SCALE>
__device__ __forceinline__ void fill_denominators(const MomView& p, double E2, double is, bool massless,
                                                  PointRec<R, N>& rec) {
    static_assert(N <= 5, "n >= 6 forms its denominators set by set (set_denominator)");
    {
        double d[N], sij[N * (N - 1) / 2 > 0 ? N * (N - 1) / 2 : 1];
#pragma unroll
        for (int i = 0; i < N; ++i) {
            const double e = p(i, 0), x = p(i, 1), y = p(i, 2), z = p(i, 3);
            d[i] = massless ? -(2.0 * E2 * (e + z)) : (e * e - x * x - y * y - z * z) - 2.0 * E2 * (e + z);
#pragma unroll
            for (int j = i + 1; j < N; ++j)
                sij[pair_index<N>(i, j)] = 2.0 * (e * p(j, 0) - x * p(j, 1) - y * p(j, 2) - z * p(j, 3));
        }
        double t[1 << (N - 1)];   // t_U for the sets U below the current highest photon
        double e[1 << (N - 1)];   // e_h(U)
#pragma unroll
        for (int h = 0; h < N; ++h) {
            e[0] = d[h];
#pragma unroll
            for (int U = 1; U < (1 << h); ++U) {
                const int l = __popc((U & -U) - 1);
                e[U] = e[U & (U - 1)] + sij[pair_index<N>(l, h)];
            }
#pragma unroll
            for (int U = 0; U < (1 << h); ++U) {
                const int T = U | (1 << h);
                if (T == (1 << N) - 1) continue;
                const double tt = U ? t[U] + e[U] : e[0];
                rec.t[T] = rec_value<R>(SCALE ? tt * is : tt);
                if (h < N - 1) t[T] = tt;
            }
        }
    }
}

// One denominator of an FP64 record for n >= 6 (one thread per set keeps
// every lane of the FP64 pipe busy): t_T = (sum_{i in T} k_i - p2)^2 by
// components, times `is` if SCALE.  Callers run it over (record, set) pairs
// after the records are built (denominators_parallel).
template <class R, int N, bool SCALE>
__device__ __forceinline__ R set_denominator(const MomView& p, double E2, double is, unsigned T) {
    double q0 = -E2, q1 = 0.0, q2 = 0.0, q3 = E2;
#pragma unroll 1
    for (int i = 0; i < N; ++i)
        if (T >> i & 1) {
            q0 += p(i, 0);
            q1 += p(i, 1);
            q2 += p(i, 2);
            q3 += p(i, 3);
        }
    const double tt = q0 * q0 - q1 * q1 - q2 * q2 - q3 * q3;
    return rec_value<R>(SCALE ? tt * is : tt);
}

// Photon sets as bitmasks: C(n, k), and the rank of S among the sets of its
// size in numeric order (numeric order of bitmasks is colexicographic order,
// so rank(S) = sum over the set bits b_1 < b_2 < ... of C(b_m, m)).
__host__ __device__ constexpr int set_binom(int n, int k) {
    if (k < 0 || k > n) return 0;
    int r = 1;
    for (int i = 1; i <= k; ++i) r = r * (n - k + i) / i;
    return r;
}
// offset of the size-k sets in a list ordered by size, then numerically
__host__ __device__ constexpr int set_level_offset(int n, int k) {
    int o = 0;
    for (int j = 0; j < k; ++j) o += set_binom(n, j);
    return o;
}
template <int N>
__device__ __forceinline__ int set_rank(unsigned S) {
    int r = 0, m = 0;
#pragma unroll
    for (int b = 0; b < N; ++b)
        if (S >> b & 1) r += set_binom(b, ++m);
    return r;
}
// list[offset(|S|) + rank(S)] = S for every S < 2^N (and rank[S] = rank(S)
// if rank != NULL), by threads lid = 0 .. nthr-1.
template <int N>
__device__ __forceinline__ void build_set_list(unsigned char* list, unsigned char* rank, int lid, int nthr) {
    for (int S = lid; S < (1 << N); S += nthr) {
        const int r = set_rank<N>((unsigned)S);
        list[set_level_offset(N, __popc(S)) + r] = (unsigned char)S;
        if (rank) rank[S] = (unsigned char)r;
    }
}

// float -> double by integer operations on the bit pattern (exact; f32_rn
// leaves no subnormals, so only zero needs its own case).
__device__ __forceinline__ double f64_of_f32(float f) {
    const unsigned int u = __float_as_uint(f);
    const unsigned int e = (u >> 23) & 0xFFu;
    const unsigned int hi = e == 0u ? (u & 0x80000000u) : (u & 0x80000000u) | ((e + 896u) << 20) | ((u & 0x7FFFFFu) >> 3);
    return __hiloint2double((int)hi, (int)(e == 0u ? 0u : u << 29));
}

// Invariant q of a record from FP64 momenta p, p1 = E1 (1, 0, 0, 1) and
// p2 = E2 (1, 0, 0, -1): q < N: d_q; N <= q < N + N(N-1)/2: s_ij for
// q = N + pair_index(i, j); after them d'_i; times `is` if SCALE.
template <int N, bool SCALE>
__device__ __forceinline__ double rec_invariant(const MomView& p, double E1, double E2, double is, bool massless,
                                                int q) {
    constexpr int NP = N * (N - 1) / 2;
    double v;
    if (q < N || q >= N + NP) {
        const bool one = q >= N + NP;   // d'_i: against p1
        const int i = one ? q - N - NP : q;
        const double e = p(i, 0), x = p(i, 1), y = p(i, 2), z = p(i, 3);
        const double lin = one ? 2.0 * E1 * (e - z) : 2.0 * E2 * (e + z);
        v = massless ? -lin : (e * e - x * x - y * y - z * z) - lin;
    } else {
        int i = 0, r = q - N;
        while (r >= N - 1 - i) {
            r -= N - 1 - i;
            ++i;
        }
        const int j = i + 1 + r;
        v = 2.0 * (p(i, 0) * p(j, 0) - p(i, 1) * p(j, 1) - p(i, 2) * p(j, 2) - p(i, 3) * p(j, 3));
    }
    return SCALE ? v * is : v;
}

// v as hi + lo: hi = v rounded to float, lo = the rest rounded to float
// (|v - hi - lo| <= 2^-48 |v| roughly).
__device__ __forceinline__ float2 split_ff(double v) {
    const float hi = f32_rn(v);
    return make_float2(hi, f32_rn(v - f64_of_f32(hi)));
}

// t_T of a record that holds invariants: their float-float sum over the
// smaller of T and its complement S (the d_i over T, or the d'_i over S,
// then the s_ij, i < j, by increasing i then j), each term added with an
// error-free two-sum into (S, E); rounded once to float.
template <int N>
__device__ __forceinline__ float rec_denominator(const float2* inv, unsigned T) {
    constexpr int NP = N * (N - 1) / 2;
    const bool comp = __popc(T) > N / 2;
    const unsigned U = comp ? ((1u << N) - 1) & ~T : T;
    const float2* lin = inv + (comp ? N + NP : 0);
    float S = 0.0f, E = 0.0f;
    auto add = [&](const float2 x) {
        const float s = S + x.x;
        const float bb = s - S;
        const float e = (S - (s - bb)) + (x.x - bb);
        S = s;
        E += e + x.y;
    };
    for (unsigned a = U; a; a &= a - 1) add(lin[__ffs(a) - 1]);
    for (unsigned a = U; a; a &= a - 1) {
        const int i = __ffs(a) - 1;
        for (unsigned b = a & (a - 1); b; b &= b - 1) add(inv[N + pair_index<N>(i, __ffs(b) - 1)]);
    }
    return S + E;
}

// 1/rs^2 of rs > 0: on the mantissa (recip_series) with the exponent put back,
// or by division where that leaves the normal range.
__device__ __forceinline__ double inverse_square(double rs) {
    const int hi = __double2hiint(rs), ex = (hi >> 20) - 1023;
    if (ex < -400 || ex > 400) return 1.0 / (rs * rs);
    const double r = recip_series(__hiloint2double(hi - (ex << 20), __double2loint(rs)));
    const double q = r * r;   // in [1/4, 1]
    return __hiloint2double(__double2hiint(q) - ((2 * ex) << 20), __double2loint(q));
}

// Record of a point that passed the cuts, from its photon momenta (units of
// EventInfo), iM and rs: momenta / sqrt(s-hat), denominators, normalisations,
// the factor to the event weight, valid = mask = 1.  The momenta are scaled
// in place, and the denominators formed from the scaled values.  (The caller
// sets idx and hsel; `fac`, the factor to |M|^2, is not needed here.)
template <class R, int N>
__device__ __forceinline__ void pass_to_rec(const MomView& v, double iM, double rs, const Physics& ph,
                                            PointRec<R, N>& rec) {
#pragma unroll 1
    for (int a = 0; a < N; ++a)
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const double k = v(a, m) * iM;
            v(a, m) = k;
            rec.k[a][m] = rec_value<R>(k);
        }
    if constexpr (N <= 5) fill_denominators<R, N, false>(v, 0.5, 1.0, true, rec);   // n >= 6: denominators_parallel
    rec.e1 = R(0.5);
    rec.e2 = R(0.5);
    rec.n1 = R(1);
    rec.n2 = R(1);
    rec.wfac = ph.wconst * inverse_square(rs);   // w = wfac * (scaled |M|^2 sum)
    rec.valid = 1;
    rec.mask = 1;
}

}  // namespace heget
