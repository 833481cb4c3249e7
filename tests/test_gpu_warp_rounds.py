"""The tree's warp rounds (n = 4, 5) at the edges of warps, rounds and tiles:
|M|^2 in FP32 and FP64 against the oracle for row counts around the rounds of
a warp, a tile and a block, with and without a helicity mask, and an invalid
row among valid ones."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [4, 5])
@pytest.mark.parametrize("N", [1, 2, 3, 5, 15, 17, 33, 47, 49, 63, 65, 130])
@pytest.mark.parametrize("tile", [0, 16, 48, 64])
def test_row_counts_around_the_rounds(oracle, heget_lib, gpu, n, N, tile):
    import torch
    H = heget_lib
    ps = oracle.phase_space(n, 0x0908440300000061, 0, N, oracle.fixed(400.0))
    mom = torch.from_numpy(ps["momenta"].copy()).cuda()
    words = max(1, (1 << (n + 2)) // 32)
    mask = torch.tensor([0x0F5A3C96 ^ (0x11111111 * w) for w in range(words)], dtype=torch.int32, device="cuda")
    for prec, tol in ((H.HEGET_FP64, 1e-10), (H.HEGET_FP32, 1e-3)):   # the tolerances of the parity tests' tails
        H.heget_set_tile(gpu, n, prec, 0, tile)
        try:
            for hm in (None, mask):
                out = torch.full((N,), -1.0, dtype=torch.float64, device="cuda")
                H.heget_amp2(gpu, n, N, mom, out, hel_mask=hm, precision=prec)
                H.heget_check(gpu)
                ref = oracle.amp2(n, ps["momenta"], hel_mask=None if hm is None else hm.cpu().numpy().view(np.uint32))
                np.testing.assert_allclose(out.cpu().numpy(), ref, rtol=tol)
        finally:
            H.heget_set_tile(gpu, n, prec, 0, 0)


@pytest.mark.parametrize("n", [4, 5])
def test_an_invalid_row_among_valid_ones(oracle, heget_lib, gpu, n):
    import torch
    H, N = heget_lib, 37
    ps = oracle.phase_space(n, 0x0908440300000062, 0, N, oracle.fixed(400.0))
    mom = torch.from_numpy(ps["momenta"].copy()).cuda()
    mom[18, 3, 1] = float("nan")
    out = torch.empty(N, dtype=torch.float64, device="cuda")
    H.heget_amp2(gpu, n, N, mom, out, precision=H.HEGET_FP32)
    with pytest.raises(H.HegetError):
        H.heget_check(gpu)
    got = out.cpu().numpy()
    assert np.isnan(got[18])
    keep = np.arange(N) != 18
    np.testing.assert_allclose(got[keep], oracle.amp2(n, ps["momenta"])[keep], rtol=1e-3)
