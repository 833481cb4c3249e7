"""heget_xsec_noalloc in FP64 at n = 4, 5, whose tiles are smaller than those
its limits are stated in: the same bits as heget_xsec_async on both sides of
4096 tiles and at the largest accepted N, one point more refused."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu

SEED = 0x09084403000000B1
TILE = {4: 96, 5: 32}
LIMIT = {4: 4096 * 128, 5: 4096 * 64}


@pytest.mark.parametrize("n", [4, 5])
def test_fp64_calls_around_4096_tiles(heget_lib, gpu, n):
    import torch
    H = heget_lib
    for N in (4096 * TILE[n], 4096 * TILE[n] + 1, 4096 * TILE[n] + 50_000, LIMIT[n]):
        for seed in (SEED, SEED + 1, SEED + 2):
            out = []
            for call in (lambda r: H.heget_xsec_async(gpu, n, seed, 0, N, H.sampler_toy_pdf(), 64, r),
                         lambda r: H.heget_xsec_noalloc(0, n, seed, 0, N, H.sampler_toy_pdf(), 64, r)):
                r = torch.zeros(80, dtype=torch.uint8, device="cuda")
                call(r)
                out.append(bytes(r.cpu().numpy()))
            assert out[0] == out[1], (N, seed)
    r = torch.zeros(80, dtype=torch.uint8, device="cuda")
    s = H.sampler_toy_pdf()
    assert H.load().heget_xsec_noalloc(0, n, 1, 0, LIMIT[n] + 1, ctypes.byref(s), None, 64, r.data_ptr(),
                                       None) == H.HEGET_EINVAL
