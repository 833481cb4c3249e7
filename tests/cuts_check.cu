// Device driver of the cut decisions (heget_ps.cuh) on momenta that the
// generator makes once in 1e16 events: prints pass_cuts_fast and pass_cuts for
// a well separated event, and for the same with its mass and momenta not
// numbers or infinite.  Compiled and run by tests/test_gpu_cuts_nan.py.
#include <cstdio>
#include <limits>

#include "heget_ps.cuh"

using namespace heget;

constexpr int kN = 2;

__global__ void decide(double* mom, const double* iM, int cases, Physics ph, int* out) {
    const int c = threadIdx.x;
    if (c >= cases) return;
    EventInfo ev{};
    ev.rs = 500.0;
    ev.iM = iM[c];
    ev.ua = ev.ub = 1ull << 52;
    const MomView v{mom + c, cases, kMomSlots};
    out[2 * c] = pass_cuts_fast<kN>(v, ev, ph);
    out[2 * c + 1] = pass_cuts<kN>(v, ev.rs * ev.iM, ev.ua, ev.ub, ph);
}

int main() {
    const double nan = std::numeric_limits<double>::quiet_NaN(), inf = std::numeric_limits<double>::infinity();
    // the components' values, 0 for the event's own, and 1/M
    const double value[] = {0, nan, -nan, inf, nan, -nan}, invm[] = {0.5, nan, -nan, inf, inf, inf};
    constexpr int kCases = 6;
    const double ev[kN][4] = {{1, 0.8, 0, 0.6}, {1, -0.8, 0, -0.6}};
    double *mom, *iM;
    int* out;
    if (cudaMallocManaged(&mom, sizeof(double) * kCases * kN * kMomSlots) || cudaMallocManaged(&iM, sizeof(double) * kCases) ||
        cudaMallocManaged(&out, sizeof(int) * 2 * kCases))
        return 1;
    for (int c = 0; c < kCases; ++c) {
        iM[c] = invm[c];
        for (int a = 0; a < kN; ++a)
            for (int m = 0; m < 4; ++m) mom[(a * kMomSlots + m) * kCases + c] = c ? value[c] : ev[a][m];
    }
    for (double pt_min : {0.0, 1.0}) {
        Physics ph{};
        ph.pt_min = pt_min;
        ph.eta_max = 2.5;
        ph.dr_min = -1.0;
        ph.sinh_eta = 6.0502044810397875;
        ph.cosh_eta = 6.1322894796636857;
        ph.cos_dr = 1.0;
        decide<<<1, 32>>>(mom, iM, kCases, ph, out);
        if (cudaDeviceSynchronize() != cudaSuccess) return 1;
        for (int c = 0; c < kCases; ++c) std::printf("%d %d\n", out[2 * c], out[2 * c + 1]);
    }
    return 0;
}
