"""heget_hist at the edges of its batches (256 events of nonzero weight) and of
its integer sums: sizes around a batch, sparse weights, weights over many
orders of magnitude, signed, infinite and NaN weights, bins so fine or so far
away that FP32 decides none of them, and energies outside the FP32 range."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def specs(H):
    return [(H.HEGET_OBS_PT_MAX, 20, 20.0, 320.0), (H.HEGET_OBS_PT, 30, 20.0, 320.0), (H.HEGET_OBS_ETA, 10, -2.5, 2.5),
            (H.HEGET_OBS_DR, 24, 0.4, 5.2), (H.HEGET_OBS_DR_MIN, 24, 0.4, 5.2), (H.HEGET_OBS_SQRT_S, 16, 100.0, 900.0)]


def run(H, gpu, n, N, w, sp, smp):
    import torch
    out = torch.empty(H.hist_bins(sp), dtype=torch.float64, device="cuda")
    H.heget_hist(gpu, n, 0x0908440300000071, 3, N, smp, torch.from_numpy(np.ascontiguousarray(w)).cuda(), sp, out)
    return out.cpu().numpy().reshape(-1, 2)


def ref(oracle, n, N, w, sp, osmp):
    ps = oracle.phase_space(n, 0x0908440300000071, 3, N, osmp)
    return np.concatenate(oracle.hist(n, ps["momenta"], ps["y"], w, sp))


def close(got, want, w):
    # bins exact; sums in integers and double-double, one rounding: against the oracle's own (compensated or plain)
    # sums a few ulp of sum |w| of the bin
    np.testing.assert_allclose(got[:, 0], want[:, 0], rtol=1e-12, atol=1e-13 * np.abs(w).max() if w.size else 0)
    np.testing.assert_allclose(got[:, 1], want[:, 1], rtol=1e-12)


@pytest.mark.parametrize("n", [2, 4, 8])
@pytest.mark.parametrize("N", [1, 255, 256, 257, 600, 1300])
def test_sizes_around_a_batch(oracle, heget_lib, gpu, n, N):
    H = heget_lib
    r = np.random.default_rng(N)
    for density in (1.0, 0.4, 0.01):
        w = r.random(N) * (r.random(N) < density)
        close(run(H, gpu, n, N, w, specs(H), H.sampler_toy_pdf()),
              ref(oracle, n, N, w, specs(H), oracle.toy_pdf()), w)


def test_weights_over_many_magnitudes_and_signs(oracle, heget_lib, gpu):
    H, n, N = heget_lib, 4, 900
    r = np.random.default_rng(4)
    w = 10.0 ** r.uniform(-40, 40, N)
    close(run(H, gpu, n, N, w, specs(H), H.sampler_toy_pdf()),
          ref(oracle, n, N, w, specs(H), oracle.toy_pdf()), np.zeros(1))
    w = r.standard_normal(N)
    close(run(H, gpu, n, N, w, specs(H), H.sampler_toy_pdf()),
          ref(oracle, n, N, w, specs(H), oracle.toy_pdf()), w)


def test_infinite_and_nan_weights_touch_their_bins_only(oracle, heget_lib, gpu):
    H, n, N = heget_lib, 3, 400
    for bad in (np.inf, np.nan):
        w = np.ones(N)
        w[[17, 300]] = bad
        got = run(H, gpu, n, N, w, specs(H), H.sampler_toy_pdf())
        touched = ref(oracle, n, N, np.where(np.isfinite(w), 0.0, 1.0), specs(H), oracle.toy_pdf())
        clean = ref(oracle, n, N, np.where(np.isfinite(w), 1.0, 0.0), specs(H), oracle.toy_pdf())
        hit = touched[:, 0] > 0
        assert not np.isfinite(got[hit]).any()
        np.testing.assert_array_equal(got[~hit], clean[~hit])


@pytest.mark.parametrize("rs", [1e-5, 500.0, 1e12])
def test_bins_that_fp32_cannot_decide(oracle, heget_lib, gpu, rs):
    """Bins far finer than FP32, and energies it does not hold: counts equal the oracle's."""
    H, n, N = heget_lib, 4, 700
    sp = [(H.HEGET_OBS_PT, 200, 0.2 * rs, 0.2 * rs * (1 + 1e-6)), (H.HEGET_OBS_PT_MAX, 50, 0.1 * rs, 0.5 * rs),
          (H.HEGET_OBS_ETA, 300, 0.5, 0.5 + 1e-5), (H.HEGET_OBS_DR, 40, 0.0, 6.0), (H.HEGET_OBS_DR_MIN, 100, 1.0, 1.0 + 1e-4)]
    w = np.ones(N)
    got = run(H, gpu, n, N, w, sp, H.sampler_fixed(rs))
    want = ref(oracle, n, N, w, sp, oracle.fixed(rs))
    np.testing.assert_array_equal(got, want)
