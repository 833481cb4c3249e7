"""The integer RAMBO momenta (csrc/heget_dir.cuh) on the host against 200-bit
values: random uniforms, the ends of (0, 1), quadrant and table boundaries,
photons along the beam, and energies next to 0."""
import os
import random
import shutil
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_0908_4403_gb300", "csrc")


def inputs():
    r = random.Random(5)
    one = 1 << 53

    def odd(x):
        return min(max(int(x), 0), one - 1) | 1
    out = [[odd(r.randrange(one)) for _ in range(4)] for _ in range(4000)]
    ends = [1, 3, one - 1, one - 3, odd(one // 2), odd(one // 2) - 2, odd(one // 4), odd(3 * one // 4) - 2]
    out += [[a, b, c, d] for a in ends for b in ends for c in ends for d in ends]
    for j in range(0, 2049):        # breakpoints of the angle, of the polar sine and of the mantissa
        x = one * j // 2048
        out.append([odd(x), odd(x), odd(one - 1), odd(x)])
        out.append([odd(x) - 2 if x > 4 else 1, odd(x) - 2 if x > 4 else 1, odd(one - 1), odd(x) - 2 if x > 4 else 1])
    for k in range(1, 53):          # small energies, small angles to the beam, small azimuths
        x = one >> k
        out.append([odd(one - x), odd(x), odd(one - x), odd(one - x)])
        out.append([odd(x), odd(one - x), odd(x), odd(x)])
    return out


def test_integer_momenta_on_the_host(tmp_path):
    mpmath = pytest.importorskip("mpmath")
    mpmath.mp.prec = 200
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not found")
    exe = tmp_path / "dir_check"
    subprocess.run([nvcc, "-std=c++17", "-O2", "--expt-relaxed-constexpr", "-gencode",
                    "arch=compute_103a,code=sm_103a", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
                    os.path.join(ROOT, "tests", "dir_check.cu"), "-o", str(exe)], check=True, capture_output=True)
    pts = inputs()
    text = "\n".join(" ".join(map(str, p)) for p in pts)
    got = subprocess.run([str(exe)], input=text, capture_output=True, text=True, check=True).stdout.split("\n")
    mp, unit = mpmath.mpf, mpmath.mpf(2) ** -53
    worst = [0.0, 0.0]
    for p, line in zip(pts, got):
        q = [float.fromhex(t) for t in line.split()]
        r = [mp(x) * unit for x in p]
        e = -mpmath.log(r[2] * r[3])
        c = 2 * r[0] - 1
        s = mpmath.sqrt(1 - c * c)
        phi = 2 * mpmath.pi * r[1]
        ref = [e, e * s * mpmath.cos(phi), e * s * mpmath.sin(phi), e * c]
        # the logarithm within 2^-62 and one rounding to FP64; the components within 2^-56 q0 more
        d = [abs(mp(a) - b) for a, b in zip(q, ref)]
        worst[0] = max(worst[0], float(d[0] / (e * mp(2) ** -53 + mp(2) ** -62)))
        for a, b in zip(d[1:], ref[1:]):
            worst[1] = max(worst[1], float(a / (abs(b) * mp(2) ** -53 + e * mp(2) ** -56 + mp(2) ** -62)))
    assert worst[0] <= 1.01 and worst[1] <= 1.01, worst


def test_committed_table_matches_its_generator(tmp_path):
    out = tmp_path / "t.h"
    subprocess.run([sys.executable, os.path.join(CSRC, "gen_dirtab.py"), str(out)], check=True)
    assert out.read_bytes() == open(os.path.join(CSRC, "heget_dirtab.h"), "rb").read()
