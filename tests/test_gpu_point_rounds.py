"""heget_amp2 in FP64 by the tree at n = 2, 3: up to 64 points of a tile
share out a point over 2^n lanes, more take a thread a point.
Every row has the same bits either way: around that line and the edges of the
warps, with and without a helicity mask, in small tiles, and beside a refused
row."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SEED = 0x0908440300000091
FULL = 300   # rows of a call whose first tile is full (256 rows at n = 2, 128 at n = 3)


def amp2(H, ctx, n, mom, mask, tile=0):
    import torch
    out = torch.full((mom.shape[0],), -1.0, dtype=torch.float64, device="cuda")
    H.heget_set_tile(ctx, n, H.HEGET_FP64, 0, tile)
    try:
        H.heget_amp2(ctx, n, mom.shape[0], mom, out, hel_mask=mask, precision=H.HEGET_FP64)
    finally:
        H.heget_set_tile(ctx, n, H.HEGET_FP64, 0, 0)
    return out.cpu().numpy()


@pytest.mark.parametrize("n", [2, 3])
@pytest.mark.parametrize("N", [1, 2, 3, 7, 15, 16, 17, 31, 32, 33, 63, 64, 65, 128])
def test_rows_of_small_calls_have_the_bits_of_full_tiles(heget_lib, gpu, n, N):
    import torch
    H = heget_lib
    mom = torch.empty(FULL, n + 2, 4, dtype=torch.float64, device="cuda")
    H.heget_phase_space_ex(gpu, SEED + n, 0, FULL, n, H.sampler_uniform(200.0, 2000.0), momenta=mom)
    mask = torch.tensor([0x0F5A3C96], dtype=torch.int32, device="cuda")
    for m in (None, mask):
        full = amp2(H, gpu, n, mom, m)
        np.testing.assert_array_equal(amp2(H, gpu, n, mom[:N].contiguous(), m), full[:N])
    for tile in (64, 128):   # (multiples of 256 / 2^n)
        np.testing.assert_array_equal(amp2(H, gpu, n, mom[:N + 64].contiguous(), None, tile), amp2(H, gpu, n, mom, None)[:N + 64])
    H.heget_check(gpu)


@pytest.mark.parametrize("n", [2, 3])
@pytest.mark.parametrize("N", [1, 5, 20, 50])
def test_a_refused_row(oracle, heget_lib, gpu, n, N):
    import torch
    from helpers import fp64_tolerance
    H = heget_lib
    ps = oracle.phase_space(n, SEED, 0, N, oracle.fixed(400.0))["momenta"]
    mom = torch.from_numpy(ps.copy()).cuda()
    mom[N // 2, 2, 1] = float("nan")
    got = amp2(H, gpu, n, mom, None)
    with pytest.raises(H.HegetError):
        H.heget_check(gpu)
    keep = np.arange(N) != N // 2
    assert np.isnan(got[N // 2])
    ref = oracle.amp2(n, ps)
    assert np.all(np.abs(got - ref)[keep] <= (fp64_tolerance(ps) * np.abs(ref))[keep])
