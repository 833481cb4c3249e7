"""Sums of squared weights in bins of small weights beside one weight many
binades above them (heget_hist adds a batch's squares as integers aligned to
the largest): within half a unit in the last place of the exact sum, plus the
rounding of the terms to 55 bits."""
import math
from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SEED, N, n = 0x09084403000000C1, 900, 4


def worst_mantissa(shift):
    """A weight just above 1 whose square loses the most below its last `shift` bits."""
    r = np.random.default_rng(3)
    return max((1.0 + float(k) * 2.0 ** -52 for k in r.integers(1, 1 << 46, 4000)),
               key=lambda w: (int(math.ldexp(w, 52)) ** 2) % (1 << shift))


@pytest.mark.parametrize("binades", [10, 27, 28, 29, 30, 31, 60])
def test_squares_beside_a_large_weight(oracle, heget_lib, gpu, binades):
    import torch
    H = heget_lib
    w0 = worst_mantissa(max(1, 2 * min(binades, 30) - 7))
    w = np.full(N, w0)
    w[450] = math.ldexp(1.5, binades)
    specs = [(H.HEGET_OBS_PT_MAX, 20, 20.0, 320.0), (H.HEGET_OBS_ETA, 10, -2.5, 2.5), (H.HEGET_OBS_DR, 24, 0.4, 5.2)]
    ps = oracle.phase_space(n, SEED, 0, N, oracle.toy_pdf())
    small, large = np.ones(N), np.zeros(N)
    small[450], large[450] = 0.0, 1.0
    c = np.concatenate(oracle.hist(n, ps["momenta"], ps["y"], small, specs))[:, 0]
    one = np.concatenate(oracle.hist(n, ps["momenta"], ps["y"], large, specs))[:, 0]
    out = torch.empty(H.hist_bins(specs), dtype=torch.float64, device="cuda")
    H.heget_hist(gpu, n, SEED, 0, N, H.sampler_toy_pdf(), torch.from_numpy(w).cuda(), specs, out)
    got = out.cpu().numpy().reshape(-1, 2)
    for b in range(len(c)):
        exact = int(c[b]) * Fraction(w0) ** 2 + int(one[b]) * Fraction(float(w[450])) ** 2
        slack = Fraction(math.ulp(float(exact))) / 2 + exact / 2 ** 55
        assert abs(Fraction(float(got[b, 1])) - exact) <= slack, (b, int(c[b]))
        exact = int(c[b]) * Fraction(w0) + int(one[b]) * Fraction(float(w[450]))
        assert abs(Fraction(float(got[b, 0])) - exact) <= Fraction(math.ulp(float(exact))) / 2 + exact / 2 ** 100
