"""The integer combination of partial sums (csrc/heget_reduce.cuh): on the
host against exact rational sums, and the device's reductions at the edges of
warps, blocks and grids through heget_sum."""
import math
import os
import random
import shutil
import subprocess
from fractions import Fraction

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def cases():
    r = random.Random(11)
    out = [[0.0], [1.0], [-1.0, 1.0], [1e300, 1e-300], [5e-324, 5e-324, -5e-324], [2.0 ** -1022, -5e-324],
           [1.7976931348623157e308], [1e16, 0.1, -1e16], [-3.0, 1e-40], [0.0, -0.0]]
    for count in (2, 31, 64, 600):
        out.append([r.uniform(0, 1) * 10.0 ** r.uniform(-12, 0) for _ in range(count)])
        out.append([r.gauss(0, 1) * 10.0 ** r.uniform(-30, 30) for _ in range(count)])
        out.append([r.uniform(-1, 1) for _ in range(count)])
    return out


def test_fixed_point_sums_on_the_host(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    exe = tmp_path / "reduce_check"
    subprocess.run([nvcc, "-std=c++17", "--expt-relaxed-constexpr", "-gencode", "arch=compute_103a,code=sm_103a",
                    "-I", os.path.join(ROOT, "include"), "-I", os.path.join(ROOT, "paper_0908_4403_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "reduce_check.cu"), "-o", str(exe)], check=True, capture_output=True)
    cs = cases() + [[1.0, math.inf], [math.nan, 1.0], [math.inf, -math.inf]]
    feed = "\n".join(f"{len(c)} " + " ".join(x.hex() for x in c) for c in cs)
    out = subprocess.run([str(exe)], input=feed, capture_output=True, text=True, check=True).stdout.split("\n")
    for c, line in zip(cs, out):
        hi, lo = (float.fromhex(t) for t in line.split())
        if not all(math.isfinite(x) for x in c):
            assert math.isnan(hi)
            continue
        exact = sum(map(Fraction, c))
        # bits dropped: each term below 2^(em - 1075 - top) (top = 73 - bits of 2 n; nothing below a subnormal's
        # last bit), and the total below 106 bits
        top = 73 - (2 * len(c)).bit_length()
        em = max(max(math.frexp(abs(x))[1] + 1022, 1) if x else 1 for x in c)
        bound = len(c) * Fraction(2) ** (em - 1075 - top) + abs(exact) / 2 ** 105 + Fraction(2) ** -1074
        assert abs(Fraction(hi) + Fraction(lo) - exact) <= bound, c[:4]


@pytest.mark.gpu
@pytest.mark.parametrize("N", [1, 31, 32, 33, 255, 257, 155649])
@pytest.mark.parametrize("kind", ["weights", "signed", "cancel"])
def test_device_sums_at_the_edges(heget_lib, gpu, N, kind):
    import numpy as np
    import torch
    r = np.random.default_rng(N)
    x = r.random(N) * 10.0 ** r.uniform(-12, 0, N)
    if kind != "weights":
        x *= r.choice([-1.0, 1.0], N)
    if kind == "cancel" and N > 2:
        x[0], x[-1] = 1e12, -1e12
    out = torch.empty(2, dtype=torch.float64, device="cuda")
    heget_lib.heget_sum(gpu, torch.from_numpy(x).cuda(), N, out)
    s, s2 = out.cpu().numpy()
    # a thread's double-double additions and the integer steps each stay below 2^-100 of sum |x|; one final rounding
    scale = math.fsum(abs(x))
    assert abs(s - math.fsum(x)) <= math.ulp(abs(math.fsum(x))) + scale * N * 2.0 ** -100
    assert abs(s2 - math.fsum(x * x)) <= math.ulp(math.fsum(x * x))


@pytest.mark.gpu
def test_device_sum_of_non_finite_values_is_nan(heget_lib, gpu):
    import torch
    out = torch.empty(2, dtype=torch.float64, device="cuda")
    for bad in (math.inf, -math.inf, math.nan):
        x = torch.ones(1000, dtype=torch.float64, device="cuda")
        x[777] = bad
        heget_lib.heget_sum(gpu, x, 1000, out)
        assert torch.isnan(out).all()
