// The integer RAMBO momenta (heget_dir.cuh) on the device: root_estimate for
// every argument against its bounds, and photon_q against the host's (which
// tests/test_dir.py holds against high-precision values) for random uniforms
// and the ends of their range.  Prints the number of violations of each.
// Compiled and run by tests/test_gpu_dir.py.
#include <cmath>
#include <cstdio>
#include <vector>

#define HEGET_DIR_TABLE static __device__ const
#include "heget_dir.cuh"

using namespace heget;
struct Words {
    u64 x, y, z, w;
};
typedef unsigned __int128 u128;

__global__ void roots(unsigned long long* bad) {
    unsigned long long n = 0;
    for (u64 x = (1ull << 30) + blockIdx.x * (u64)blockDim.x + threadIdx.x; x < (1ull << 32);
         x += (u64)gridDim.x * blockDim.x) {
        const u64 Y = root_estimate((u32)x);
        // Y 2^-30 <= 1 / sqrt(x 2^-32) at the upper end, and above (1 - 2^-20) of it at the lower one
        const u128 sq = (u128)Y * Y, one = (u128)1 << 92;
        n += sq * (x + 1) > one || sq * x < one - (one >> 19);
    }
    if (n) atomicAdd(bad, n);
}

__global__ void momenta(const Words* r, PhotonQ* q, int n) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        q[i] = photon_q(r[i].x, r[i].y, r[i].z, r[i].w, kDirLog, kDirAng);
}

int main() {
    unsigned long long* bad;
    if (cudaMallocManaged(&bad, sizeof *bad)) return 1;
    *bad = 0;
    roots<<<1024, 256>>>(bad);
    if (cudaDeviceSynchronize() != cudaSuccess) return 1;
    std::printf("root_estimate %llu\n", *bad);

    const u64 one = 1ull << 53, ends[] = {1, 3, one - 1, one - 3, one / 2 + 1, one / 2 - 1, one / 4 + 1, 3 * (one / 4) - 1};
    std::vector<Words> in;
    for (u64 a : ends)
        for (u64 b : ends)
            for (u64 c : ends)
                for (u64 d : ends) in.push_back(Words{a, b, c, d});
    u64 s = 1;
    auto next = [&] { return (s = s * 6364136223846793005ull + 1442695040888963407ull) >> 11 | 1; };
    for (int i = 0; i < 1000000; ++i) in.push_back(Words{next(), next(), next(), next()});
    for (int k = 1; k < 53; ++k)   // towards the beam and small energies
        for (int j = 0; j < 200; ++j)
            in.push_back(Words{next() >> k | 1, next(), one - (next() >> k | 1) | 1, one - (next() >> k | 1) | 1});
    const int n = (int)in.size();
    Words* r;
    PhotonQ* q;
    if (cudaMallocManaged(&r, n * sizeof *r) || cudaMallocManaged(&q, n * sizeof *q)) return 1;
    for (int i = 0; i < n; ++i) r[i] = in[i];
    momenta<<<1024, 128>>>(r, q, n);
    if (cudaDeviceSynchronize() != cudaSuccess) return 1;
    // the tables for the host's side
    static uint4 logtab[kDirTable];
    static ulonglong2 angtab[kDirTable];
    if (cudaMemcpyFromSymbol(logtab, kDirLog, sizeof logtab) || cudaMemcpyFromSymbol(angtab, kDirAng, sizeof angtab)) return 1;
    int off = 0;
    for (int i = 0; i < n; ++i) {
        const PhotonQ h = photon_q(r[i].x, r[i].y, r[i].z, r[i].w, logtab, angtab);
        // each side within q0 2^-56 + 2^-62 of the true value and one rounding
        const double slack = 2 * (h.q0 * 0x1p-56 + 0x1p-62);
        auto near = [&](double a, double b) { return std::fabs(a - b) <= slack + std::fabs(b) * 0x1p-52; };
        off += !(q[i].q0 == h.q0 && near(q[i].q1, h.q1) && near(q[i].q2, h.q2) && near(q[i].q3, h.q3));
    }
    std::printf("photon_q %d of %d\n", off, n);
    return 0;
}
