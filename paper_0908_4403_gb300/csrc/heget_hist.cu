// heget_hist.cu -- kinematic distributions (Sec. 5, Fig. 2): weighted
// histograms of photon observables of the generated events.  The events of
// nonzero weight are regenerated from the counter-based generator, 256 at a
// time; their bins come from FP32 observables wherever FP32 settles them, and
// the weights are added as integers within a batch (w exactly, w^2 rounded to
// 55 bits or more a term) and in double-double across batches and blocks, in a
// fixed order, so results are reproducible bit for bit for a given launch shape
// (one resident wave, set by the GPU).
//
// What bounded the earlier form (GB300, five histograms of 1,048,576 events at
// n = 4: 5480 us): 2690 FP64 instruction slots an event -- the observables'
// asinh, atan2, log and square roots in FP64, bin sums with one active lane an
// FP64 instruction, and the events of zero weight, generated and dropped.
// Here, 97 slots (41 % of the FP64 pipe) and 154 warp instructions an event: 511
// us, bound by the barriers between the passes of a batch (six a histogram).
#include <algorithm>
#include <cmath>

#include "heget_kernels.cuh"
#include "heget_internal.h"

namespace heget {
namespace {

constexpr int kHistBlock = 256;   // events of a batch, one per thread

struct HistSpecDev {
    int kind, nbins, off, pad;   // off: first bin of this histogram in the block's bin array
    double lo, scale;            // scale = nbins / (hi - lo), formed on the host
    float lo_f, scale_f;
};

struct HistArgs {
    HistSpecDev spec[HEGET_HIST_MAX_SPECS];
    int nspec, total, most;   // bins of all histograms, of the largest
};

// Bin of x: 0 below lo (and NaN), nbins + 1 at or above hi, else
// 1 + floor((x - lo) scale), in FP64 without contraction.
__device__ __forceinline__ int hist_bin(double x, int nbins, double lo, double scale) {
    if (!(x >= lo)) return 0;
    const double t = __dmul_rn(__dsub_rn(x, lo), scale);
    if (t >= (double)nbins) return nbins + 1;
    return 1 + (int)t;
}

constexpr float kHistU = 5.9604645e-8f;   // 2^-24

// The same bin from an FP32 value xf of x, |xf - x| <= err: -1 unless the bin
// is certain.  (x - lo) scale carries err scale, the roundings of lo and of the
// difference (4 u |lo|, u |xf|) and 4 u of itself; every bin edge is an integer.
__device__ __forceinline__ int hist_bin_f(float xf, float err, const HistSpecDev& h) {
    const float t = (xf - h.lo_f) * h.scale_f;
    const float d = (err + 4.0f * kHistU * (fabsf(h.lo_f) + fabsf(xf))) * h.scale_f + 4.0f * kHistU * fabsf(t);
    const float nb = (float)h.nbins;
    if (t < -d) return 0;
    if (t > nb + d) return h.nbins + 1;
    if (fabsf(t - rintf(t)) > d) return t < nb ? 1 + (int)t : -1;
    return -1;   // next to an edge, or not a number
}

__host__ __device__ constexpr int hist_entries_max(int n) {
    return n * (n - 1) / 2 > n ? n * (n - 1) / 2 : n;
}

// Shared memory of a block: momenta; the weights as integers (w, w^2); the
// entries (bin, place in it) and the events sorted by bin; counts and offsets
// per bin; bin sums of w and w^2; sampler draws; the list of events.
struct HistFixed {
    __int128 w, w2;
};
__host__ __device__ constexpr size_t hist_smem_bytes(int n, int total, int most) {
    return (size_t)n * kMomSlots * kHistBlock * sizeof(double) + kHistBlock * sizeof(HistFixed) +
           2 * (size_t)total * sizeof(DD) + kHistBlock * sizeof(SampleDraw) +
           2 * kHistBlock * (sizeof(long long) + sizeof(double)) +
           (size_t)hist_entries_max(n) * kHistBlock * (sizeof(unsigned) + sizeof(unsigned char)) +
           2 * (size_t)most * sizeof(unsigned);
}

// One event's observables in FP64, for the bins that FP32 leaves open.
struct HistEvent {
    MomView v;
    double scale, y;
    __device__ __forceinline__ double pt(int i) const {
        const double px = v(i, 1) * scale, py = v(i, 2) * scale;
        return sqrt(__dadd_rn(__dmul_rn(px, px), __dmul_rn(py, py)));
    }
    __device__ __forceinline__ double eta(int i) const { return asinh(v(i, 3) * scale / pt(i)) + y; }
    __device__ __forceinline__ double dr(int a, int b) const {
        double dphi = fabs(atan2(v(a, 2) * scale, v(a, 1) * scale) - atan2(v(b, 2) * scale, v(b, 1) * scale));
        if (dphi > M_PI) dphi = 2.0 * M_PI - dphi;
        const double deta = eta(a) - eta(b);
        return sqrt(__dadd_rn(__dmul_rn(deta, deta), __dmul_rn(dphi, dphi)));
    }
};
// Observable `kind` of photon i or pair (i, j) (or the event's extreme) in FP64, binned.
template <int N>
__device__ __noinline__ int hist_bin_exact(const MomView v, double scale, u64 ua, u64 ub, int i, int j, int kind,
                                           int nbins, double lo, double per_unit) {
    EventInfo ev;
    ev.ua = ua;
    ev.ub = ub;
    const HistEvent e{v, scale, ua == ub ? 0.0 : event_rapidity(ev)};
    double x = 0.0;
    if (kind == HEGET_OBS_PT) x = e.pt(i);
    else if (kind == HEGET_OBS_ETA) x = e.eta(i);
    else if (kind == HEGET_OBS_DR) x = e.dr(i, j);
    else if (kind == HEGET_OBS_PT_MAX) {
        x = e.pt(0);
        for (int a = 1; a < N; ++a) x = e.pt(a) > x ? e.pt(a) : x;
    } else {
        x = e.dr(0, 1);
        for (int a = 0; a < N; ++a)
            for (int b = a + 1; b < N; ++b) {
                const double d = e.dr(a, b);
                x = d < x ? d : x;
            }
    }
    return hist_bin(x, nbins, lo, per_unit);
}

// (Three blocks an SM up to n = 5: 85 registers.)
template <int N>
__global__ void __launch_bounds__(kHistBlock, N <= 5 ? 3 : 1)
hist_kernel(uint64_t seed, long long i0, long long npts, SamplerArgs S, Physics ph,
            const double* __restrict__ w, HistArgs H, double* __restrict__ parts) {
    constexpr int NP = N * (N - 1) / 2, NW = kHistBlock / 32;
    constexpr int E = hist_entries_max(N);
    // w: terms below 2^(53 + kTop); w^2: products of mantissas below 2^(106 + kTop2); a bin has at most
    // E kHistBlock < 2^13 terms of a batch.  The least w^2 of a pass, 2^104 2^(kTop2 - 2 kSpan), keeps 55 bits
    constexpr int kTop = 60, kTop2 = 7, kSpan = 28;
    extern __shared__ __align__(16) unsigned char smem[];
    HistFixed* fx = reinterpret_cast<HistFixed*>(smem);
    SampleDraw* draws = reinterpret_cast<SampleDraw*>(fx + kHistBlock);
    DD* hw = reinterpret_cast<DD*>(draws + kHistBlock);
    DD* hw2 = hw + H.total;
    double* stage = reinterpret_cast<double*>(hw2 + H.total);
    long long* list = reinterpret_cast<long long*>(stage + (size_t)N * kMomSlots * kHistBlock);   // events to come
    double* lw = reinterpret_cast<double*>(list + 2 * kHistBlock);                                // their weights
    unsigned* ent = reinterpret_cast<unsigned*>(lw + 2 * kHistBlock);   // [entry][event]: bin | place << 10
    unsigned* cnt = ent + E * kHistBlock;
    unsigned* off = cnt + H.most;
    unsigned char* sorted = reinterpret_cast<unsigned char*>(off + H.most);
    HistFixed* bin_sum = reinterpret_cast<HistFixed*>(draws);
    __shared__ int s_cnt[NW];
    __shared__ unsigned s_em[NW];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    for (int b = tid; b < H.total; b += kHistBlock) hw[b] = hw2[b] = DD{0.0, 0.0};
    const MomView v{stage + tid, kHistBlock, kMomSlots};
    long long t0 = (long long)blockIdx.x * kHistBlock;
    int ln = 0;   // events in the list
    while (t0 < npts || ln > 0) {
        // the next events of nonzero weight, in order (a zero weight adds nothing)
        while (ln < kHistBlock && t0 < npts) {
            const long long i = t0 + tid;
            const double wi = i < npts ? w[i] : 0.0;
            int tot;
            const int pos = compact_pos<kHistBlock>(wi != 0.0, tid, s_cnt, 0, tot);
            if (wi != 0.0) {
                list[ln + pos] = i0 + i;
                lw[ln + pos] = wi;
            }
            ln += tot;
            t0 += (long long)gridDim.x * kHistBlock;
        }
        __syncthreads();
        const int cur = min(ln, kHistBlock);
        // sampler draws by two warps, 128 events each
        if (warp < 2 && cur > warp * (kHistBlock / 2)) {
            const int b0 = warp * (kHistBlock / 2);
            warp_draws(S, seed, [&](int p) { return (uint64_t)list[b0 + p]; }, min(cur - b0, kHistBlock / 2), draws + b0);
        }
        __syncthreads();
        EventInfo ev;
        ev.ua = ev.ub = 1;
        ev.rs = 0.0;
        double wi = 0.0, scale = 0.0;
        float pt[N], eta[N], phi[N], yf = 0.0f;
        bool fp32 = false;   // FP32 holds the event
        if (tid < cur) {
            sample_finish(S, draws[tid], ev);
            ev.iM = rambo<N>(PointRng(seed, (uint64_t)list[tid]), v);
            scale = ev.rs * ev.iM;
            wi = lw[tid];
            fp32 = fp32_holds(ev);
            const float sf = f32_cut(fp32 ? scale : 0.0);
            // errors (u = 2^-24, components 2 u): pT 10 u; eta = ln((E + |pz|) / pT) 16 u absolute and 2 u of
            // itself; phi 16 u absolute; y = ln(ua / ub) 10 u absolute and 2 u of itself
#pragma unroll
            for (int i = 0; i < N; ++i) {
                const float e = f32_cut(v(i, 0)), x = f32_cut(v(i, 1)), y = f32_cut(v(i, 2)), z = f32_cut(v(i, 3));
                const float p2 = x * x + y * y, rp = rsqrtf(p2);
                pt[i] = p2 * rp * sf;
                eta[i] = copysignf(logf((e + fabsf(z)) * rp), z);
                phi[i] = atan2f(y, x);
                fp32 = fp32 && p2 > 1e-30f;
            }
            if (ev.ua != ev.ub) yf = logf(__fdividef(__ull2float_rn(ev.ua), __ull2float_rn(ev.ub)));
        }
        // the rest of the list moves up
        long long keep_i = 0;
        double keep_w = 0.0;
        if (cur + tid < ln) {
            keep_i = list[cur + tid];
            keep_w = lw[cur + tid];
        }
        __syncthreads();
        if (cur + tid < ln) {
            list[tid] = keep_i;
            lw[tid] = keep_w;
        }
        ln -= cur;
        // passes over the batch: the events whose weights lie within 2^kSpan of the largest left, as integers
        // aligned to it (almost always all of them); infinite and NaN weights make their bins NaN
        bool left = tid < cur;
        for (;;) {
            const int ef = left ? exponent_field(wi) : 0;
            const unsigned wm = __reduce_max_sync(0xffffffffu, (unsigned)ef);
            if (lane == 0) s_em[warp] = wm;
            __syncthreads();
            int em = 0;
#pragma unroll
            for (int q = 0; q < NW; ++q) em = max(em, (int)s_em[q]);
            if (em == 0) break;
            const bool mine = left && (em >= 0x7FF ? ef == em : ef >= em - kSpan);
            left = left && !mine;
            if (mine && em < 0x7FF) {
                const u64 u = double_bits(wi);
                const int f = (int)(u >> 52) & 0x7FF;
                const u64 m = (u & 0xFFFFFFFFFFFFFull) | (f ? 1ull << 52 : 0ull);
                const unsigned __int128 m2 = (unsigned __int128)m * m;
                const int sh = kTop2 - 2 * (em - ef);
                fx[tid].w = fixed_of(wi, em, kTop);
                fx[tid].w2 = (__int128)(sh >= 0 ? m2 << sh : (m2 + ((unsigned __int128)1 << (-sh - 1))) >> -sh);
            }
            for (int s = 0; s < H.nspec; ++s) {
                const HistSpecDev& h = H.spec[s];
                const int nb = h.nbins + 2;
                for (int b = tid; b < nb; b += kHistBlock) cnt[b] = 0;
                __syncthreads();   // (also: the integers above, s_em read)
                int m = 0;
                if (mine) {
                    auto put = [&](int bin) {
                        ent[m * kHistBlock + tid] = (unsigned)bin | (atomicAdd(cnt + bin, 1u) << 10);
                        ++m;
                    };
                    auto exact = [&](int i, int j) { 
                        return hist_bin_exact<N>(v, scale, ev.ua, ev.ub, i, j, h.kind, h.nbins, h.lo, h.scale);
                    };
                    if (h.kind == HEGET_OBS_PT_MAX || h.kind == HEGET_OBS_PT) {
                        float mx = pt[0];
#pragma unroll
                        for (int i = 0; i < N; ++i) {
                            mx = fmaxf(mx, pt[i]);
                            if (h.kind == HEGET_OBS_PT) {
                                const int b = fp32 ? hist_bin_f(pt[i], 12.0f * kHistU * pt[i], h) : -1;
                                put(b >= 0 ? b : exact(i, 0));
                            }
                        }
                        if (h.kind == HEGET_OBS_PT_MAX) {
                            const int b = fp32 ? hist_bin_f(mx, 12.0f * kHistU * mx, h) : -1;
                            put(b >= 0 ? b : exact(0, 0));
                        }
                    } else if (h.kind == HEGET_OBS_ETA) {
#pragma unroll
                        for (int i = 0; i < N; ++i) {
                            const float x = eta[i] + yf;
                            const int b =
                                fp32 ? hist_bin_f(x, kHistU * (32.0f + 4.0f * (fabsf(eta[i]) + fabsf(yf))), h) : -1;
                            put(b >= 0 ? b : exact(i, 0));
                        }
                    } else if (h.kind == HEGET_OBS_DR || h.kind == HEGET_OBS_DR_MIN) {
                        float dmin = 3.0e38f, emin = 0.0f;   // smallest Delta R, largest error
#pragma unroll
                        for (int a = 0; a < N; ++a)
#pragma unroll
                            for (int b = a + 1; b < N; ++b) {
                                float dphi = fabsf(phi[a] - phi[b]);
                                if (dphi > 3.14159265f) dphi = 6.28318531f - dphi;
                                const float deta = eta[a] - eta[b];
                                const float dr = sqrtf(deta * deta + dphi * dphi);
                                const float err = kHistU * (80.0f + 4.0f * (fabsf(eta[a]) + fabsf(eta[b])));
                                if (h.kind == HEGET_OBS_DR) {
                                    const int q = fp32 ? hist_bin_f(dr, err, h) : -1;
                                    put(q >= 0 ? q : exact(a, b));
                                }
                                dmin = fminf(dmin, dr);
                                emin = fmaxf(emin, err);
                            }
                        if (h.kind == HEGET_OBS_DR_MIN) {
                            const int q = fp32 ? hist_bin_f(dmin, emin, h) : -1;
                            put(q >= 0 ? q : exact(0, 1));
                        }
                    } else {
                        put(hist_bin(ev.rs, h.nbins, h.lo, h.scale));
                    }
                }
                __syncthreads();
                // offsets of the bins in the sorted list
                if (warp == 0) {
                    unsigned run = 0;
                    for (int b0 = 0; b0 < nb; b0 += 32) {
                        const unsigned c = b0 + lane < nb ? cnt[b0 + lane] : 0u;
                        unsigned x = c;
#pragma unroll
                        for (int o = 1; o < 32; o <<= 1) {
                            const unsigned y = __shfl_up_sync(0xffffffffu, x, o);
                            if (lane >= o) x += y;
                        }
                        if (b0 + lane < nb) off[b0 + lane] = run + x - c;
                        run += __shfl_sync(0xffffffffu, x, 31);
                    }
                }
                __syncthreads();
                for (int e = 0; e < m; ++e) {
                    const unsigned q = ent[e * kHistBlock + tid];
                    sorted[off[q & 1023u] + (q >> 10)] = (unsigned char)tid;
                }
                __syncthreads();
                // bin sums: the order of a bin's events is that of the counting, but integer sums do not depend
                // on it; 2^ls lanes share a bin
                int ls = 0;
                while (ls < 5 && (nb << (ls + 1)) <= kHistBlock) ++ls;
                for (int q0 = 0; q0 < (nb << ls); q0 += kHistBlock) {
                    const int b = (q0 + tid) >> ls, part = tid & ((1 << ls) - 1);
                    __int128 a = 0, a2 = 0;
                    unsigned c = 0;
                    if (b < nb) {
                        c = cnt[b];
                        const unsigned char* o = sorted + off[b];
                        if (em < 0x7FF)
                            for (unsigned q = part; q < c; q += 1u << ls) {
                                a += fx[o[q]].w;
                                a2 += fx[o[q]].w2;
                            }
                    }
                    for (int o = (1 << ls) >> 1; o > 0; o >>= 1) {
                        a += shfl_down128(a, o);
                        a2 += shfl_down128(a2, o);
                    }
                    // the sums go to one thread a bin, so that the FP64 additions below run with whole warps (the
                    // room of the sampler draws: at most 128 bins are shared)
                    if (ls > 0) {
                        if (part == 0 && b < nb) bin_sum[b] = HistFixed{a, a2};
                        __syncthreads();
                        if (tid < nb) {
                            a = bin_sum[tid].w;
                            a2 = bin_sum[tid].w2;
                            c = cnt[tid];
                        }
                    }
                    const int mb = ls > 0 ? tid : b;
                    if (mb < nb && c > 0) {
                        DD *d = hw + h.off + mb, *d2 = hw2 + h.off + mb;
                        if (em < 0x7FF) {
                            *d = dd_add(*d, dd_of_int(a, em - 1075 - kTop));
                            *d2 = dd_add(*d2, dd_of_int(a2, 2 * (em - 1075) - kTop2));
                        } else {
                            *d = *d2 = DD{bits_double(0x7FF8000000000000ull), 0.0};
                        }
                    }
                }
                __syncthreads();
            }
        }
        __syncthreads();   // the momenta and s_em are free again
    }
    __syncthreads();
    for (int b = tid; b < H.total; b += kHistBlock) {
        double* o = parts + ((size_t)blockIdx.x * H.total + b) * 4;
        o[0] = hw[b].hi;
        o[1] = hw[b].lo;
        o[2] = hw2[b].hi;
        o[3] = hw2[b].lo;
    }
}

// Block partials of a bin combined by one warp, as integers aligned to the
// largest exponent (heget_reduce.cuh), into out[2b], out[2b + 1].  (GB300, 608
// blocks, 234 bins: 57 us as two kernels of double-double additions.)
__global__ void __launch_bounds__(256) hist_finalize_kernel(const double* __restrict__ parts, int nblocks, int total,
                                                            double* __restrict__ out) {
    const int b = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (b >= total) return;
    int em[2] = {1, 1};
    for (int k = lane; k < nblocks; k += 32) {
        const double* o = parts + ((size_t)k * total + b) * 4;
        em[0] = max(em[0], exponent_field(DD{o[0], o[1]}));
        em[1] = max(em[1], exponent_field(DD{o[2], o[3]}));
    }
    const int top = 73 - (32 - __clz(2 * nblocks));   // 2 nblocks terms below 2^(53 + top)
    __int128 v[2] = {0, 0};
#pragma unroll
    for (int q = 0; q < 2; ++q) em[q] = (int)__reduce_max_sync(0xffffffffu, (unsigned)em[q]);
    for (int k = lane; k < nblocks; k += 32) {
        const double* o = parts + ((size_t)k * total + b) * 4;
        v[0] += fixed_of(DD{o[0], o[1]}, em[0], top);
        v[1] += fixed_of(DD{o[2], o[3]}, em[1], top);
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        for (int o = 16; o > 0; o >>= 1) v[q] += shfl_down128(v[q], o);
        if (lane == 0) {
            const DD d = dd_of_fixed(v[q], em[q], top);
            out[2 * b + q] = d.hi + d.lo;
        }
    }
}

template <int N>
int launch_hist_n(uint64_t seed, long long i0, long long npts, const SamplerArgs& S, const Physics& ph,
                  const double* w, const HistArgs& H, double* parts, int grid, cudaStream_t st) {
    auto k = hist_kernel<N>;
    const size_t smem = hist_smem_bytes(N, H.total, H.most);
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return (int)e;
    k<<<grid, kHistBlock, smem, st>>>(seed, i0, npts, S, ph, w, H, parts);
    return (int)cudaGetLastError();
}

template <int N>
int occupancy_hist_n(int total, int most, int* bpsm) {
    auto k = hist_kernel<N>;
    const size_t smem = hist_smem_bytes(N, total, most);
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return (int)e;
    return (int)cudaOccupancyMaxActiveBlocksPerMultiprocessor(bpsm, k, kHistBlock, smem);
}

}  // namespace
}  // namespace heget

using namespace heget;

extern "C" {

int heget_hist(heget_ctx* ctx, int n, uint64_t seed, int64_t i0, int64_t N, const heget_sampler* smp,
               const double* w, const heget_hist_spec* specs, int nspec, double* out, void* stream) {
    int r = check_common(ctx, n, N);
    if (r) return r;
    if ((r = check_sampler(smp))) return r;
    if ((r = check_range(i0, N))) return r;
    if (!specs || nspec < 1 || nspec > HEGET_HIST_MAX_SPECS)
        return fail(HEGET_EINVAL, "need 1 <= nspec <= %d histogram specs", HEGET_HIST_MAX_SPECS);
    HistArgs H{};
    H.nspec = nspec;
    int total = 0;
    for (int s = 0; s < nspec; ++s) {
        const heget_hist_spec& q = specs[s];
        if (q.observable < HEGET_OBS_PT_MAX || q.observable > HEGET_OBS_SQRT_S)
            return fail(HEGET_EINVAL, "spec %d: unknown observable %d", s, q.observable);
        if (q.nbins < 1 || q.nbins > HEGET_HIST_MAX_BINS - 2)
            return fail(HEGET_EINVAL, "spec %d: nbins = %d", s, q.nbins);
        if (!std::isfinite(q.lo) || !std::isfinite(q.hi) || !(q.lo < q.hi) || !std::isfinite(q.hi - q.lo) ||
            !std::isfinite((double)q.nbins / (q.hi - q.lo)))
            return fail(HEGET_EINVAL, "spec %d: need finite lo < hi and a finite bins-per-unit scale", s);
        H.spec[s].kind = q.observable;
        H.spec[s].nbins = q.nbins;
        H.spec[s].off = total;
        H.spec[s].lo = q.lo;
        H.spec[s].scale = (double)q.nbins / (q.hi - q.lo);
        H.spec[s].lo_f = (float)H.spec[s].lo;
        H.spec[s].scale_f = (float)H.spec[s].scale;
        total += q.nbins + 2;
        H.most = std::max(H.most, q.nbins + 2);
    }
    if (total > HEGET_HIST_MAX_BINS) return fail(HEGET_EINVAL, "%d bins in all; at most %d", total, HEGET_HIST_MAX_BINS);
    H.total = total;
    if (!out) return fail(HEGET_EINVAL, "out must be non-NULL");
    if (N > 0 && !w) return fail(HEGET_EINVAL, "w must be non-NULL");
    DeviceGuard g(ctx->device);
    cudaStream_t st = (cudaStream_t)stream;
    if (N == 0) {
        const cudaError_t e = cudaMemsetAsync(out, 0, 2 * (size_t)total * sizeof(double), st);
        return e == cudaSuccess ? HEGET_OK : cuda_fail(e, "heget_hist");
    }
    int bpsm = 0;
#define OCC(NN) occupancy_hist_n<NN>(total, H.most, &bpsm)
    switch (n) {
        case 2: r = OCC(2); break;
        case 3: r = OCC(3); break;
        case 4: r = OCC(4); break;
        case 5: r = OCC(5); break;
        case 6: r = OCC(6); break;
        case 7: r = OCC(7); break;
        default: r = OCC(8); break;
    }
#undef OCC
    if (r) return cuda_fail((cudaError_t)r, "hist occupancy");
    // one resident wave of at most four blocks per SM keeps the block partials few
    const long long tiles = (N + kHistBlock - 1) / kHistBlock;
    const long long wave = (long long)ctx->num_sms * std::min(std::max(bpsm, 1), 4);
    const int grid = (int)std::min(tiles, wave);
    const size_t part_bytes = (size_t)grid * total * 4 * sizeof(double);
    if ((r = grow((void**)&ctx->hist_parts, &ctx->hist_parts_cap, part_bytes, false))) return r;
    const SamplerArgs S = sampler_args(smp);
    const Physics ph = physics_of(ctx, n);
#define RUN(NN) launch_hist_n<NN>(seed, i0, N, S, ph, w, H, ctx->hist_parts, grid, st)
    switch (n) {
        case 2: r = RUN(2); break;
        case 3: r = RUN(3); break;
        case 4: r = RUN(4); break;
        case 5: r = RUN(5); break;
        case 6: r = RUN(6); break;
        case 7: r = RUN(7); break;
        default: r = RUN(8); break;
    }
#undef RUN
    if (r) return cuda_fail((cudaError_t)r, "hist_kernel");
    hist_finalize_kernel<<<(total + 7) / 8, 256, 0, st>>>(ctx->hist_parts, grid, total, out);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return cuda_fail(e, "hist_finalize_kernel");
    return HEGET_OK;
}

}  // extern "C"
