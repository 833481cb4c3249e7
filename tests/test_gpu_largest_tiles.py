"""The largest tiles of the fused FP32 subset recursion: 314 points at n = 7 and
270 at n = 8 fill a block's shared memory to 32 and 64 bytes; the next ones are
refused by the launch."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,tile,step", [(7, 314, 2), (8, 270, 1)])
def test_the_largest_tiles_run(heget_lib, gpu, n, tile, step):
    import torch
    H, N, s = heget_lib, 700, heget_lib.sampler_toy_pdf()
    H.heget_set_algorithm(gpu, H.HEGET_ALG_SUBSET)
    out = {}
    try:
        for t in (64, tile):
            H.heget_set_tile(gpu, n, 32, 1, t)
            w = torch.empty(N, dtype=torch.float64, device="cuda")
            res = torch.zeros(80, dtype=torch.uint8, device="cuda")
            H.heget_xsec_async(gpu, n, 5, 0, N, s, 32, res, w_out=w)
            out[t] = w.cpu().numpy(), H.result_from_tensor(res)
        H.heget_set_tile(gpu, n, 32, 1, tile + step)
        with pytest.raises(H.HegetError):
            H.heget_xsec_async(gpu, n, 5, 0, N, s, 32, res, w_out=w)
    finally:
        H.heget_set_tile(gpu, n, 32, 1, 0)
        H.heget_set_algorithm(gpu, H.HEGET_ALG_TREE)
    np.testing.assert_array_equal(out[tile][0], out[64][0])
    assert out[tile][1].n_pass == out[64][1].n_pass > 0
    np.testing.assert_allclose(out[tile][1].sum_w, out[64][1].sum_w, rtol=1e-15)
