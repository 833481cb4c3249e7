"""The warp-specialised subset kernel (n = 7, 8) around the edges of its
producers' stages (96 and 64 events), its consumer groups and its grid: every
weight in FP32 against the FP64 kernel."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SEED = 0x0908440300000071


@pytest.mark.parametrize("n", [7, 8])
@pytest.mark.parametrize("N", [1, 63, 64, 65, 95, 96, 97, 129, 193, 64 * 152 + 1, 96 * 152 + 1])
def test_counts_around_the_stages(heget_lib, gpu, n, N):
    import torch
    H = heget_lib
    H.heget_set_algorithm(gpu, H.HEGET_ALG_SUBSET)
    try:
        w, tot = {}, {}
        for prec in (H.HEGET_FP32, H.HEGET_FP64):
            out = torch.full((N,), -1.0, dtype=torch.float64, device="cuda")
            res = torch.zeros(80, dtype=torch.uint8, device="cuda")
            H.heget_xsec_async(gpu, n, SEED, 7, N, H.sampler_uniform(500.0, 2000.0), prec, res, out)
            H.heget_check(gpu)
            w[prec], tot[prec] = out.cpu().numpy(), H.result_from_tensor(res)
    finally:
        H.heget_set_algorithm(gpu, H.HEGET_ALG_TREE)
    # the cut decisions do not depend on the precision of the amplitudes
    np.testing.assert_array_equal(w[H.HEGET_FP32] == 0, w[H.HEGET_FP64] == 0)
    np.testing.assert_allclose(w[H.HEGET_FP32], w[H.HEGET_FP64], rtol=1e-3)   # the parity tests' tail
    assert tot[H.HEGET_FP32].n_pass == tot[H.HEGET_FP64].n_pass == np.count_nonzero(w[H.HEGET_FP64])
