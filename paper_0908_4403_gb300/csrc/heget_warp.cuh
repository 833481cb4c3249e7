// heget_warp.cuh -- amplitude rounds of the ordering tree at n = 4 and 5, one
// configuration per lane, by whole warps on their own: the same orderings, products and order of additions as
// tree_amplitude (heget_amp.cuh), bit for bit.
//
// What bounded the lane-by-lane walk: issue slots and block barriers, not the
// FMA pipe.  Every lane recomputed the row after the first two (three)
// photons for its own helicities, although the row depends on those photons'
// helicities only -- 4 (8) values shared by 16 (32) lanes -- and each step
// cost table index arithmetic of its own; the block met at four barriers a
// round.  Here the rows of every ordered prefix are formed once per helicity
// assignment of the prefix (R2: 12 x 4 rows at n = 4; at n = 5 R2: 20 x 4, R3:
// 60 x 8 in chunks of one first photon), and the lanes only close them with
// the pair columns of the two photons left: 24 (120) closures a lane, their
// table offsets known at compile time up to the lane's helicity bits.  The
// phases of a warp's points are separated by warp barriers.
//
// GB300, warp instructions a point and time, walk -> here: the n = 4 step of
// 1,048,576 points 661 -> 384 and 1027 -> 644 us (its consumers were what the FP64
// producers waited for); heget_amp2 of 50,001 rows at n = 5 5013 -> 2500 and 322 ->
// 190 us; FP64 at n = 4, 262,144 points 3030 -> 2346 us, and 1806 with the orders
// of a pair added first (warp_add_orders).  (These rounds alone; with the
// sampler's warp and the FP64 tiles the calls take 611, 187 and 1587 us.)  What
// bounds it now: fixed latencies and the instruction cache (issue 51 %, FMA pipe
// 31 %, FP64 pipe 47 % of the fused n = 4 kernel).
#pragma once

#include "heget_amp.cuh"

namespace heget {

template <class R, int N, int HB>
__host__ __device__ constexpr bool tree_warp_rounds() {
    return HB == 0 && (N == 4 || N == 5) && tree_two_ended<R, N>();
}

// E = eps*(k, lambda) . sigma = [[e00, e01], [e10, -e00]] of a photon: its
// entries as step_matrix forms them, e00, e01, Re e10 in a row, Im e10 apart.
template <class R>
struct EHel {
    Row<R> a;
    R e10i;
};
template <class R>
__device__ __forceinline__ EHel<R> e_of(const Row<R>& ph, int lam_bit) {
    const R rs2 = R(0.70710678118654752440);
    const R lam = lam_bit ? R(1) : R(-1);
    const R am = fmad<R>(-lam, ph.ai, R(1)) * rs2, ap = fmad<R>(lam, ph.ai, R(1)) * rs2;
    return EHel<R>{Row<R>{-lam * ph.ar * rs2, -am * ph.br, am * ph.bi, ap * ph.br}, ap * ph.bi};
}

// The same from a momentum, with 1 -+ lambda cos theta formed from k_z and 1/|k|
// in one rounding (FP64 at n = 2, 3); every fused operation written out, so
// that results have the same bits wherever it is inlined.
template <class R>
struct PhotonDir {
    R z, rk, st, cp, sp;   // k_z, 1/|k|, sin theta, cos phi, sin phi
};
template <class R>
__device__ __forceinline__ PhotonDir<R> photon_dir(const R* k) {
    const R pt2 = fmad<R>(k[1], k[1], k[2] * k[2]), ka2 = fmad<R>(k[3], k[3], pt2);
    PhotonDir<R> d{k[3], rsq<R>(ka2), R(0), R(1), R(0)};   // (a photon along z: as photon_row)
    if (pt2 > R(1e-24) * ka2) {
        const R rpt = rsq<R>(pt2);
        d.st = pt2 * rpt * d.rk;
        d.cp = k[1] * rpt;
        d.sp = k[2] * rpt;
    }
    return d;
}
template <class R>
__device__ __forceinline__ EHel<R> e_of(const PhotonDir<R>& d, int lam_bit) {
    const R rs2 = R(0.70710678118654752440);
    const R lam = lam_bit ? R(1) : R(-1);
    const R am = fmad<R>(-lam * d.z, d.rk, R(1)) * rs2, ap = fmad<R>(lam * d.z, d.rk, R(1)) * rs2;
    return EHel<R>{Row<R>{-lam * d.st * rs2, -am * d.cp, am * d.sp, ap * d.cp}, ap * d.sp};
}

// step_matrix (of E and a set) and row_times with every fused operation
// written out: the ones that the compiler makes of the plain forms in the
// lane-by-lane walk, so that results have the walk's bits whatever the code
// around.
template <class R>
struct Mat2 {
    Row<R> m0, m1;
};
template <class R>
__device__ __forceinline__ Mat2<R> step_fused(const EHel<R>& e, const Row<R>& sd) {
    const R e00 = e.a.ar, e11 = -e00, e01r = e.a.ai, e01i = e.a.br, e10r = e.a.bi, e10i = e.e10i;
    const R A = sd.ar, D = sd.ai, Br = sd.br, Bi = sd.bi;
    Mat2<R> o;
    o.m0.ar = fmad<R>(-e01i, Bi, fmad<R>(e00, A, e01r * Br));
    o.m0.ai = fmad<R>(e01i, Br, e01r * Bi);
    o.m0.br = fmad<R>(e01r, D, e00 * Br);
    o.m0.bi = fmad<R>(e01i, D, e11 * Bi);
    o.m1.ar = fmad<R>(e10r, A, e11 * Br);
    o.m1.ai = fmad<R>(e10i, A, e11 * Bi);
    o.m1.br = fmad<R>(e11, D, fmad<R>(e10r, Br, e10i * Bi));
    o.m1.bi = fmad<R>(e10i, Br, -(e10r * Bi));
    return o;
}
template <class R>
__device__ __forceinline__ Row<R> row_times_fused(const Row<R>& r, const Row<R>& m0, const Row<R>& m1) {
    Row<R> o;
    o.ar = fmad<R>(-r.bi, m1.ai, fmad<R>(r.br, m1.ar, fmad<R>(r.ar, m0.ar, -(r.ai * m0.ai))));
    o.ai = fmad<R>(r.bi, m1.ar, fmad<R>(r.br, m1.ai, fmad<R>(r.ai, m0.ar, r.ar * m0.ai)));
    o.br = fmad<R>(-r.bi, m1.bi, fmad<R>(r.br, m1.br, fmad<R>(r.ar, m0.br, -(r.ai * m0.bi))));
    o.bi = fmad<R>(r.bi, m1.br, fmad<R>(r.br, m1.bi, fmad<R>(r.ai, m0.br, r.ar * m0.bi)));
    return o;
}

// Points of a warp's round: at n = 4 four where the block has at most four
// such warps (eight lanes form each point's tables: 8 (photon, helicity)
// items, 24 row and 24 column items, so that every lane has one), two with
// more warps, to leave room for two blocks an SM; one at n = 5.  The closures
// take 2^n lanes a point, PW points at a time.
__host__ __device__ constexpr int warp_round_points(int n, int warps) { return n == 5 ? 1 : warps <= 4 ? 4 : 2; }

template <class R, int N, int WARPS>
struct WarpTables {
    static constexpr int NS = 1 << N;
    static constexpr int PB = warp_round_points(N, WARPS);   // points of a round
    static constexpr int LP = 32 / PB;                  // lanes a point in the table phases
    static constexpr int PW = 32 / NS;                  // points at a time in the closures
    static constexpr int NP = N * (N - 1);              // ordered pairs
    static constexpr int NC3 = N == 5 ? (N - 1) * (N - 2) : 0;   // ordered (j2, j3) after a first photon
    // rows of a point; an odd number spreads the points over the banks
    static constexpr int PT = (8 * N + NS + 4 * NP + 4 * NP + 8 * NC3) | 1;
    static constexpr size_t bytes = (size_t)WARPS * PB * PT * sizeof(Row<R>);
    Row<R>* SD;   // [2^N]: set data
    Row<R>* EA;   // [N][2]: E of photon and helicity
    R* EI;        // [N][2], in 2 N rows' room: Im e10
    Row<R>* R1;   // [N][2]: first rows
    Row<R>* CL;   // [N][2]: closures
    Row<R>* R2;   // [ordered (j1, j2)][place2]: rows after two photons; place2: the lower photon's helicity + 2 the other's
    Row<R>* PC;   // [ordered (a, b)][place2]: pair columns
    Row<R>* R3;   // [ordered (j2, j3)][lambda_1 + 2 place2]: rows after three photons, first photon j1 (n = 5)
    __device__ __forceinline__ WarpTables(unsigned char* smem, int point) {
        SD = reinterpret_cast<Row<R>*>(smem) + (size_t)point * PT;
        EA = SD + NS;
        EI = reinterpret_cast<R*>(EA + 2 * N);
        R1 = EA + 4 * N;
        CL = R1 + 2 * N;
        R2 = CL + 2 * N;
        PC = R2 + 4 * NP;
        R3 = PC + 4 * NP;
    }
    __device__ __forceinline__ EHel<R> e(int x) const { return EHel<R>{ld_row(EA + x), EI[x]}; }
    static __device__ __forceinline__ EHel<R> make_e(const R* k, int lam_bit) { return e_of<R>(photon_row<R>(k), lam_bit); }
};

// ordered pair k = a (n - 1) + b - [b > a]
template <int N>
__device__ __forceinline__ void pair_of_slot(int k, int& a, int& b) {
    a = k / (N - 1);
    const int t = k - a * (N - 1);
    b = t + (t >= a);
}

// Tables of one point by its LP lanes (l), in three phases separated by warp
// barriers, which the caller places: E and set data; first rows and closures;
// rows after two photons and pair columns.
template <class R, int N, class WT>
__device__ __forceinline__ void warp_sets(const WT& tb, const PointRec<R, N>& rc, int l) {
    if (l < 2 * N) {
        const EHel<R> e = WT::make_e(rc.k[l >> 1], l & 1);
        st_row(tb.EA + l, e.a);
        tb.EI[l] = e.e10i;
    }
#pragma unroll 1
    for (int T = 1 + l; T < (1 << N) - 1; T += WT::LP) st_row(tb.SD + T, set_row<R, N>(rc, (unsigned)T));
}

template <class R, int N, class WT>
__device__ __forceinline__ void warp_ends(const WT& tb, const PointRec<R, N>& rc, int l) {
    if (l < 2 * N) {   // photon l / 2, helicity l % 2
        const EHel<R> e = tb.e(l);
        const Row<R> m1 = step_fused(e, ld_row(tb.SD + (1 << (l >> 1)))).m1;
        const R n1 = rc.n1, n2 = rc.n2;
        st_row(tb.CL + l, Row<R>{n1 * e.a.ar, R(0), n1 * e.a.bi, n1 * e.e10i});
        st_row(tb.R1 + l, Row<R>{n2 * m1.ar, n2 * m1.ai, n2 * m1.br, n2 * m1.bi});
    }
}

// rows after two photons: items (ordered (j1, j2), helicity of j2)
template <class R, int N, class WT>
__device__ __forceinline__ void warp_rows(const WT& tb, int l) {
    constexpr int LP = WT::LP, NI = 2 * N * (N - 1);
#pragma unroll 1
    for (int it = l; it < NI; it += LP) {
        const int lam = it & 1, k = it >> 1;
        int x, y;
        pair_of_slot<N>(k, x, y);
        const Mat2<R> m = step_fused(tb.e(2 * y + lam), ld_row(tb.SD + ((1 << x) | (1 << y))));
        const Row<R>* src = tb.R1 + 2 * x;
        Row<R>* dst = tb.R2 + 4 * k + (x < y ? lam << 1 : lam);
        const Row<R> o0 = row_times_fused(ld_row(src), m.m0, m.m1), o1 = row_times_fused(ld_row(src + 1), m.m0, m.m1);
        st_row(dst, o0);
        st_row(dst + (x < y ? 1 : 2), o1);
    }
}

template <class R, int N, int WARPS>
__device__ __forceinline__ void warp_pairs(const WarpTables<R, N, WARPS>& tb, int l) {
    constexpr int LP = WarpTables<R, N, WARPS>::LP, NI = 2 * N * (N - 1);
    constexpr unsigned FULL = (1u << N) - 1;
    warp_rows<R, N>(tb, l);
    // pair columns: items (ordered (a, b), helicity of a)
#pragma unroll 1
    for (int it = l; it < NI; it += LP) {
        const int lam = it & 1, k = it >> 1;
        int x, y;
        pair_of_slot<N>(k, x, y);
        const Mat2<R> m = step_fused(tb.e(2 * x + lam), ld_row(tb.SD + (FULL & ~(1u << y))));
        const Row<R>* src = tb.CL + 2 * y;
        Row<R>* dst = tb.PC + 4 * k + (x < y ? lam : lam << 1);
#pragma unroll
        for (int b = 0; b < 2; ++b) {
            const Row<R> c = ld_row(src + b);
            Row<R> pc{R(0), R(0), R(0), R(0)};
            close_row(m.m0, c, pc.ar, pc.ai);
            close_row(m.m1, c, pc.br, pc.bi);
            st_row(dst + (b ? (x < y ? 2 : 1) : 0), pc);
        }
    }
}

// n = 5: rows after three photons with first photon j1, items (ordered (j2,
// j3), helicity of j3), each for the four helicities of (j1, j2).
template <class R, int N, int WARPS>
__device__ __forceinline__ void warp_triples(const WarpTables<R, N, WARPS>& tb, int j1, int l) {
    constexpr int NI = 2 * (N - 1) * (N - 2);
#pragma unroll 1
    for (int it = l; it < NI; it += WarpTables<R, N, WARPS>::LP) {
        const int lam = it & 1, q = it >> 1;
        int j2, j3;
        pair_of_slot<N - 1>(q, j2, j3);   // among the photons other than j1
        j2 += j2 >= j1;
        j3 += j3 >= j1;
        const Mat2<R> sm = step_fused(tb.e(2 * j3 + lam), ld_row(tb.SD + ((1 << j1) | (1 << j2) | (1 << j3))));
        const Row<R>* src = tb.R2 + 4 * pair_slot<N>(j1, j2);
        // place in R3: helicity of j1, then those of the other two, lower photon first
        Row<R>* dst = tb.R3 + 8 * q + (j2 < j3 ? lam << 2 : lam << 1);
#pragma unroll
        for (int m = 0; m < 4; ++m) {
            const int l1 = m & 1, l2 = m >> 1;
            st_row(dst + l1 + (j2 < j3 ? l2 << 1 : l2 << 2),
                   row_times_fused(ld_row(src + (j1 < j2 ? l1 | (l2 << 1) : l2 | (l1 << 1))), sm.m0, sm.m1));
        }
    }
}

// FP64: the rows of the two orders of a photon pair and the pair columns of
// the two orders of the pair left are added first (distributivity), so that a
// set of two photons closes once instead of four times: 48 multiply-adds a
// lane at n = 4 instead of 192, where the FP64 pipe is what bounds the rounds.
// (FP32 keeps the walk's order of additions, and so its bits.)  In place, to
// the entries with the lower photon first; `rows`: R2 too (n = 4).
template <class R, int N, int WARPS>
__device__ __forceinline__ void warp_add_orders(const WarpTables<R, N, WARPS>& tb, int l, bool rows) {
    constexpr int LP = WarpTables<R, N, WARPS>::LP, NU = N * (N - 1) / 2;
    for (int it = l; it < (rows ? 8 : 4) * NU; it += LP) {
        Row<R>* t = it < 4 * NU ? tb.PC : tb.R2;
        const int q = it < 4 * NU ? it : it - 4 * NU;
        int x, y;
        pair_of_unit<N>(q >> 2, x, y);
        Row<R>* d = t + 4 * pair_slot<N>(x, y) + (q & 3);
        const Row<R> a = ld_row(d), b = ld_row(t + 4 * pair_slot<N>(y, x) + (q & 3));
        st_row(d, Row<R>{a.ar + b.ar, a.ai + b.ai, a.br + b.br, a.bi + b.bi});
    }
}

// The same contract as amplitude_rounds_lanes; BLOCK threads, whole warps.
// With BAR = 0 the block meets once at the end; the consumers of a
// warp-specialised block (BAR != 0) meet their producers right after, and the
// tables are each warp's own, so they need no barrier here.
template <class R, int N, int BLOCK, int BAR>
__device__ __forceinline__ void amplitude_rounds_warps(unsigned char* table_smem, PointRec<R, N>* recs, int cnt,
                                                       const uint32_t* mask) {
    using WT = WarpTables<R, N, BLOCK / 32>;
    constexpr int NS = WT::NS, PB = WT::PB, PW = WT::PW, LP = WT::LP, NW = BLOCK / 32;
    constexpr unsigned FULL = NS - 1;
    constexpr bool kAdd = sizeof(R) != sizeof(float);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned char* mem = table_smem + (size_t)warp * (WT::bytes / NW);
    const WT tb(mem, lane / LP);
    const int l = lane % LP;
    const unsigned h = (unsigned)(lane % NS);
    const float wh = lane_weight<N>(mask, h);
    // places of the helicities of photons x < y in this lane's configuration
    auto o2 = [&](int x, int y) { return (int)((h >> x & 1u) | ((h >> y & 1u) << 1)); };
    // sum over the lanes of |A_h|^2 w_h of point pt
    auto finish = [&](R ar, R ai, int pt) {
        // a sampled helicity (PointRec::hsel): only the selected lane counts
        const bool active = pt < cnt && recs[pt].valid;
        const int hsel = active ? recs[pt].hsel : -1;
        R v = active ? norm2(ar, ai) * R(sel_weight<N>(hsel, h, wh)) : R(0);
#pragma unroll
        for (int off = 1; off < NS; off <<= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        if (pt < cnt && h == 0) recs[pt].ssum = v;
    };
    for (int base = warp * PB; base < cnt; base += NW * PB) {
        const int p = base + lane / LP;
        const bool mine = p < cnt;
        if (mine) warp_sets(tb, recs[p], l);
        __syncwarp();
        if (mine) warp_ends(tb, recs[p], l);
        __syncwarp();
        if (mine) warp_pairs(tb, l);
        __syncwarp();
        if constexpr (kAdd) {
            // (at n = 5 the rows after two photons are extended one by one, so only the columns are added)
            if (mine) warp_add_orders(tb, l, N == 4);
            __syncwarp();
        }
        if constexpr (N == 4) {
            // (rolled over the point groups: written out side by side for more
            // independent chains it ran 4 % slower, and so did the table phases
            // unrolled, 5 %: the block's code already strains the instruction cache)
#pragma unroll 1
            for (int s = 0; s < PB / PW; ++s) {
                if (base + s * PW >= cnt) break;
                const WT tc(mem, s * PW + lane / NS);
                R ar = R(0), ai = R(0);
#pragma unroll
                for (int k = 0; k < WT::NP; ++k) {
                    const int j1 = k / (N - 1), t = k - j1 * (N - 1), j2 = t + (t >= j1);
                    if (kAdd && j1 > j2) continue;
                    const unsigned rem = FULL & ~((1u << j1) | (1u << j2));
                    const int a = __ffs(rem) - 1, b = __ffs(rem & (rem - 1)) - 1;
                    const int o = j1 < j2 ? o2(j1, j2) : o2(j2, j1);
                    const Row<R> r = ld_row(tc.R2 + 4 * k + o);
                    close_row(r, ld_row(tc.PC + 4 * pair_slot<N>(a, b) + o2(a, b)), ar, ai);
                    if (!kAdd) close_row(r, ld_row(tc.PC + 4 * pair_slot<N>(b, a) + o2(a, b)), ar, ai);
                }
                finish(ar, ai, base + s * PW + lane / NS);
            }
        } else {
            // a point at a time (PW = 1); the triples of one first photon j1 for all points together
            R are[PB], aim[PB];
#pragma unroll
            for (int s = 0; s < PB; ++s) are[s] = aim[s] = R(0);
#pragma unroll 1
            for (int j1 = 0; j1 < N; ++j1) {
                if (mine) warp_triples(tb, j1, l);
                __syncwarp();
                // the other photons by position 0 .. 3 (increasing): their helicity bits, and for each pair of
                // positions the offsets of its two pair columns
                const unsigned h1 = h >> j1 & 1u, ho = (h & ((1u << j1) - 1u)) | (h >> (j1 + 1) << j1);
                int po[6][2], k = 0;
#pragma unroll
                for (int x = 0; x < N - 1; ++x)
#pragma unroll
                    for (int y = x + 1; y < N - 1; ++y, ++k) {
                        const int a = x + (x >= j1), b = y + (y >= j1), o = (int)((ho >> x & 1u) | ((ho >> y & 1u) << 1));
                        po[k][0] = 4 * pair_slot<N>(a, b) + o;
                        po[k][1] = 4 * pair_slot<N>(b, a) + o;
                    }
#pragma unroll
                for (int s = 0; s < PB; ++s) {
                    const WT tc(mem, s);
                    const Row<R>* r3 = tc.R3 + h1;
#pragma unroll
                    for (int q = 0; q < WT::NC3; ++q) {
                        // positions (x, y) attached in this order, a < b left
                        const int x = q / (N - 2), t = q - x * (N - 2), y = t + (t >= x);
                        const unsigned rem = 15u & ~((1u << x) | (1u << y));
                        const int a = __ffs(rem) - 1, b = __ffs(rem & (rem - 1)) - 1, u = pair_index<N - 1>(a, b);
                        const int lo = x < y ? x : y, hi = x < y ? y : x;
                        const Row<R> r = ld_row(r3 + 8 * q + ((ho >> lo & 1u) << 1 | (ho >> hi & 1u) << 2));
                        close_row(r, ld_row(tc.PC + po[u][0]), are[s], aim[s]);
                        if (!kAdd) close_row(r, ld_row(tc.PC + po[u][1]), are[s], aim[s]);
                    }
                }
                __syncwarp();
            }
#pragma unroll
            for (int s = 0; s < PB; ++s) finish(are[s], aim[s], base + s);
        }
        __syncwarp();
    }
    if constexpr (BAR == 0) __syncthreads();
}

// ---------------------------------------------------------------------------
// FP64 at n = 2, 3: one thread per point.
//
// With 4 or 8 helicity configurations a point, the rounds' phases cost more
// than their work: four block barriers for 64 or 32 points, table items of
// three kinds, lanes that hold one configuration each -- some 600 FP64 slots a
// point at n = 2 for about 230 operations.  One thread forms a point's
// polarisations, rows and closures in registers and adds up all its
// configurations: every lane busy, no shared memory and no barrier.
// GB300, before -> after: 65,536 points at fixed energy 82 -> 68 us (n = 2), toy
// PDF 256 -> 212 us (n = 3).  (FP32 keeps the rounds: written this way its
// results differ in the last bit, for 10 to 20 % less time.)
// ---------------------------------------------------------------------------
template <class R, int N, int HB>
__host__ __device__ constexpr bool tree_point_rounds() {
    return sizeof(R) != sizeof(float) && HB == 0 && N <= 3;
}

template <class R, int N>
__device__ __forceinline__ R point_sum(const PointRec<R, N>& rc, const uint32_t* mask) {
    constexpr int NS = 1 << N;
    EHel<R> e[N][2];
#pragma unroll
    for (int j = 0; j < N; ++j) {
        const PhotonDir<R> d = photon_dir<R>(rc.k[j]);
        e[j][0] = e_of<R>(d, 0);
        e[j][1] = e_of<R>(d, 1);
    }
    const R n1 = rc.n1, n2 = rc.n2;
    R are[NS], aim[NS];
#pragma unroll
    for (int h = 0; h < NS; ++h) are[h] = aim[h] = R(0);
    auto closure = [&](int j, int l) {
        return Row<R>{n1 * e[j][l].a.ar, R(0), n1 * e[j][l].a.bi, n1 * e[j][l].e10i};
    };
#pragma unroll
    for (int j1 = 0; j1 < N; ++j1) {
        Row<R> r1[2];
        const Row<R> sd = set_row<R, N>(rc, 1u << j1);
#pragma unroll
        for (int l = 0; l < 2; ++l) {
            const Row<R> m1 = step_fused(e[j1][l], sd).m1;
            r1[l] = Row<R>{n2 * m1.ar, n2 * m1.ai, n2 * m1.br, n2 * m1.bi};
        }
        if constexpr (N == 2) {
#pragma unroll
            for (int h = 0; h < NS; ++h)
                close_row(r1[h >> j1 & 1], closure(1 - j1, h >> (1 - j1) & 1), are[h], aim[h]);
        } else {
#pragma unroll
            for (int t = 0; t < N - 1; ++t) {
                const int j2 = t + (t >= j1), j3 = 3 - j1 - j2;
                const Row<R> sd2 = set_row<R, N>(rc, (1u << j1) | (1u << j2));
#pragma unroll
                for (int l2 = 0; l2 < 2; ++l2) {
                    const Mat2<R> m = step_fused(e[j2][l2], sd2);
#pragma unroll
                    for (int l1 = 0; l1 < 2; ++l1) {
                        const Row<R> r2 = row_times_fused(r1[l1], m.m0, m.m1);
#pragma unroll
                        for (int l3 = 0; l3 < 2; ++l3) {
                            const int h = (l1 << j1) | (l2 << j2) | (l3 << j3);
                            close_row(r2, closure(j3, l3), are[h], aim[h]);
                        }
                    }
                }
            }
        }
    }
    R v[NS];
#pragma unroll
    for (int h = 0; h < NS; ++h)
        v[h] = norm2(are[h], aim[h]) * R(sel_weight<N>(rc.hsel, (unsigned)h, lane_weight<N>(mask, (unsigned)h)));
#pragma unroll
    for (int off = 1; off < NS; off <<= 1)
#pragma unroll
        for (int h = 0; h < NS; h += 2 * off) v[h] += v[h + off];
    return v[0];
}

// heget_amp2, up to kFewPoints points of a tile: the FP64 pipe takes as long for
// one lane as for 32, and a lane with all configurations holds it for some 1500
// instructions at n = 3.  2^n lanes of a warp share a point: tables by item as
// at n = 4, then a lane a configuration to close them; the same operations in
// the same order as point_sum, so the same bits, whatever the row count.
// GB300, heget_amp2, one thread a point -> here: n = 3, 1 to 16 rows 51 -> 16 us,
// 32 rows 52 -> 24, 64 rows 53 -> 39; n = 2, 1 row 14.6 -> 10.4, 64 rows 14.4 -> 13.4.
// With more points than a block has such warps for, one thread a point is
// ahead (the fused kernels' tiles are full, or share the SM with others).
constexpr int kFewPoints = 64;

template <class R, int N>
struct FewTables {
    static constexpr int NS = 1 << N, LP = NS;
    static constexpr int PB = 32 / LP, NW = 8;   // points of a warp, warps
    static constexpr int PT = (NS + 7 * N + (N == 3 ? 4 * N * (N - 1) : 0)) | 1;   // rows of a point
    static constexpr size_t bytes = (size_t)NW * PB * PT * sizeof(Row<R>);
    Row<R>*SD, *EA, *R1, *CL, *R2;   // as in WarpTables
    R* EI;
    __device__ __forceinline__ FewTables(unsigned char* smem, int point) {
        SD = reinterpret_cast<Row<R>*>(smem) + (size_t)point * PT;
        EA = SD + NS;
        EI = reinterpret_cast<R*>(EA + 2 * N);
        R1 = EA + 3 * N;
        CL = R1 + 2 * N;
        R2 = CL + 2 * N;
    }
    __device__ __forceinline__ EHel<R> e(int x) const { return EHel<R>{ld_row(EA + x), EI[x]}; }
    static __device__ __forceinline__ EHel<R> make_e(const R* k, int lam_bit) { return e_of<R>(photon_dir<R>(k), lam_bit); }
};

template <class R, int N, int BLOCK>
__device__ __forceinline__ void amplitude_rounds_few(unsigned char* table_smem, PointRec<R, N>* recs, int cnt,
                                                     const uint32_t* mask) {
    using FT = FewTables<R, N>;
    constexpr int LP = FT::LP, PB = FT::PB, NW = FT::NW;
    static_assert((N == 2 || N == 3) && BLOCK / 32 >= NW, "n = 2, 3");
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, l = lane % LP;
    if (warp < NW) {
        const FT tb(table_smem, warp * PB + lane / LP);
        const float wh = lane_weight<N>(mask, (unsigned)l);
        for (int base = warp * PB; base < cnt; base += NW * PB) {
            const int c = base + lane / LP;
            const bool mine = c < cnt && recs[c].valid;
            if (mine) warp_sets<R, N>(tb, recs[c], l);
            __syncwarp();
            if (mine) warp_ends<R, N>(tb, recs[c], l);
            __syncwarp();
            if constexpr (N == 3) {
                if (mine) warp_rows<R, N>(tb, l);
                __syncwarp();
            }
            R v = R(0);
            if (mine) {
                R ar = R(0), ai = R(0);
                auto bit = [&](int j) { return l >> j & 1; };
#pragma unroll
                for (int j1 = 0; j1 < N; ++j1) {
                    if constexpr (N == 2) {
                        const int j2 = 1 - j1;
                        close_row(ld_row(tb.R1 + 2 * j1 + bit(j1)), ld_row(tb.CL + 2 * j2 + bit(j2)), ar, ai);
                    } else {
#pragma unroll
                        for (int t = 0; t < N - 1; ++t) {
                            const int j2 = t + (t >= j1), j3 = 3 - j1 - j2;
                            const int o = j1 < j2 ? bit(j1) | bit(j2) << 1 : bit(j2) | bit(j1) << 1;
                            close_row(ld_row(tb.R2 + 4 * (j1 * (N - 1) + t) + o), ld_row(tb.CL + 2 * j3 + bit(j3)), ar, ai);
                        }
                    }
                }
                v = norm2(ar, ai) * R(sel_weight<N>(recs[c].hsel, (unsigned)l, wh));
            }
#pragma unroll
            for (int off = 1; off < LP; off <<= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
            if (c < cnt && l == 0) recs[c].ssum = v;
            __syncwarp();
        }
    }
    __syncthreads();
}

// The same contract as amplitude_rounds_lanes.
template <class R, int N, int BLOCK, int BAR>
__device__ __forceinline__ void amplitude_rounds_points(PointRec<R, N>* recs, int cnt, const uint32_t* mask) {
    for (int c = threadIdx.x; c < cnt; c += BLOCK) recs[c].ssum = recs[c].valid ? point_sum<R, N>(recs[c], mask) : R(0);
    if constexpr (BAR == 0) __syncthreads();
}

}  // namespace heget
