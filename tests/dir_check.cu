// Host driver of the integer RAMBO momenta (heget_dir.cuh): reads lines of
// four odd 53-bit integers, prints q0 .. q3 as hex doubles.  Compiled and run
// by tests/test_dir.py; no GPU needed.
#include <cstdio>

#define HEGET_DIR_TABLE static const
#include "heget_dir.cuh"

int main() {
    unsigned long long r[4];
    while (std::scanf("%llu %llu %llu %llu", r, r + 1, r + 2, r + 3) == 4) {
        const heget::PhotonQ q = heget::photon_q(r[0], r[1], r[2], r[3], heget::kDirLog, heget::kDirAng);
        std::printf("%a %a %a %a\n", q.q0, q.q1, q.q2, q.q3);
    }
    return 0;
}
