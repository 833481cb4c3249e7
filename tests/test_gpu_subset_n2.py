"""heget_amp2 with the subset recursion at n = 2, whose one-photon currents
come straight from the records: row counts around a round (16 points in FP32,
8 in FP64), a tile and a block, with and without a helicity mask, a photon
along the beam, and a refused row among valid ones, against the oracle."""
import numpy as np
import pytest

from helpers import fp64_tolerance

pytestmark = pytest.mark.gpu

SEED = 0x0908440300000081
U32 = 2.0 ** -24


@pytest.fixture
def subset(heget_lib, gpu):
    heget_lib.heget_set_algorithm(gpu, heget_lib.HEGET_ALG_SUBSET)
    yield gpu
    heget_lib.heget_set_algorithm(gpu, heget_lib.HEGET_ALG_TREE)


def amp2(H, ctx, mom, prec, mask=None, tile=0):
    import torch
    N = mom.shape[0]
    out = torch.full((N,), -1.0, dtype=torch.float64, device="cuda")
    m = None if mask is None else torch.from_numpy(mask.view(np.int32)).cuda()
    H.heget_set_tile(ctx, 2, prec, 0, tile)
    try:
        H.heget_amp2(ctx, 2, N, torch.from_numpy(np.ascontiguousarray(mom)).cuda(), out, hel_mask=m, precision=prec)
    finally:
        H.heget_set_tile(ctx, 2, prec, 0, 0)
    return out.cpu().numpy()


@pytest.mark.parametrize("N", [1, 7, 8, 9, 15, 16, 17, 255, 256, 257, 600])
@pytest.mark.parametrize("tile", [0, 64])
def test_row_counts_around_the_rounds(oracle, heget_lib, subset, N, tile):
    H = heget_lib
    ps = oracle.phase_space(2, SEED, 0, 4 * N + 16, oracle.fixed(400.0))
    mom = ps["momenta"][np.asarray(ps["mask"]).astype(bool)][:N].copy()   # rows that pass the cuts: no cancellations
    assert len(mom) == N
    # (masks that keep a helicity whose amplitude does not vanish: lambda_1 != lambda_2)
    for mask in (None, np.array([0xA5A5], dtype=np.uint32), np.array([0x0060], dtype=np.uint32)):
        ref = oracle.amp2(2, mom, hel_mask=mask)
        got = amp2(H, subset, mom, H.HEGET_FP64, mask, tile)
        assert np.all(np.abs(got - ref) <= fp64_tolerance(mom) * np.abs(ref))
        # some 30 roundings of FP32 on the longest path to an amplitude, squared
        got = amp2(H, subset, mom, H.HEGET_FP32, mask, tile)
        assert np.all(np.abs(got - ref) <= 64 * U32 * np.abs(ref))
    H.heget_check(subset)


def test_a_refused_row_and_a_photon_along_the_beam(oracle, heget_lib, subset):
    H = heget_lib
    mom = oracle.phase_space(2, SEED + 1, 0, 33, oracle.fixed(400.0))["momenta"].copy()
    mom[5, 2] = [200.0, 2e-9, 0.0, 200.0]     # |M|^2 finite: the propagator is not zero in FP64
    mom[5, 3] = [200.0, -2e-9, 0.0, -200.0]
    mom[20, 2, 1] = np.nan
    keep = (np.arange(33) != 20) & (np.arange(33) != 5)
    ref = oracle.amp2(2, mom[keep])
    for prec in (H.HEGET_FP64, H.HEGET_FP32):
        got = amp2(H, subset, mom, prec)
        with pytest.raises(H.HegetError):
            H.heget_check(subset)
        assert np.isnan(got[20])
        tree = None
        H.heget_set_algorithm(subset, H.HEGET_ALG_TREE)
        tree = amp2(H, subset, mom, prec)
        with pytest.raises(H.HegetError):
            H.heget_check(subset)
        H.heget_set_algorithm(subset, H.HEGET_ALG_SUBSET)
        # the collinear row: whatever the tree makes of it, to the precision's rounding
        np.testing.assert_allclose(got[5], tree[5], rtol=1e-10 if prec == H.HEGET_FP64 else 64 * U32)
        tol = fp64_tolerance(mom[keep]) if prec == H.HEGET_FP64 else 1e-3   # (no cuts here: the parity tests' tail)
        assert np.all(np.abs(got[keep] - ref) <= tol * np.abs(ref))
