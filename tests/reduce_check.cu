// Host driver of the integer combination of partial sums (heget_reduce.cuh):
// reads lines "count x1 x2 ..." of hex doubles, adds them as fixed-point
// integers aligned to the largest exponent, prints the double-double as two
// hex doubles.  Compiled and run by tests/test_reduce.py; no GPU needed.
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "heget_reduce.cuh"

using namespace heget;

int main() {
    int n;
    char buf[64];
    while (std::scanf("%d", &n) == 1) {
        std::vector<double> x(n);
        for (auto& v : x) {
            if (std::scanf("%63s", buf) != 1) return 1;
            v = std::strtod(buf, nullptr);
        }
        int em = 1, bits = 0;
        for (double v : x) em = exponent_field(v) > em ? exponent_field(v) : em;
        while ((1 << bits) <= 2 * n) ++bits;
        const int top = 73 - bits;
        __int128 s = 0;
        for (double v : x) s += fixed_of(DD{v, 0.0}, em, top);
        const DD r = dd_of_fixed(s, em, top);
        std::printf("%a %a\n", r.hi, r.lo);
    }
    return 0;
}
