"""The fused FP64 subset recursion from n = 6 on holds fewer records than a
tile generates: with cuts that every point passes, tiles of one record less
than, exactly, and more than one and two chunks of them.  Every weight has the
bits of a tile that needs one chunk only, and follows heget_amp2 of the same
events; also around the point count where n = 8 changes its default tile."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SEED = 0x09084403000000A1
CHUNK = {6: 32, 7: 24, 8: 16}


@pytest.fixture
def open_cuts(heget_lib, gpu):
    H = heget_lib
    H.heget_set_params(gpu, pt_min=0.0, eta_max=100.0, dr_min=-1.0)
    H.heget_set_algorithm(gpu, H.HEGET_ALG_SUBSET)
    yield gpu
    H.heget_set_algorithm(gpu, H.HEGET_ALG_TREE)
    H.heget_set_params(gpu)


def weights(H, ctx, n, N, tile, smp, batch=False):
    import torch
    w = torch.full((N,), -1.0, dtype=torch.float64, device="cuda")
    res = torch.zeros(80, dtype=torch.uint8, device="cuda")
    H.heget_set_tile(ctx, n, H.HEGET_FP64, 1, tile)
    try:
        if batch:
            H.heget_xsec_batch(ctx, [dict(n=n, precision=64, seed=SEED, N=N, sampler=smp, result_dev=res, w_out=w)])
        else:
            H.heget_xsec_async(ctx, n, SEED, 0, N, smp, H.HEGET_FP64, res, w_out=w)
    finally:
        H.heget_set_tile(ctx, n, H.HEGET_FP64, 1, 0)
    return w.cpu().numpy(), H.result_from_tensor(res)


@pytest.mark.parametrize("n", [6, 7, 8])
@pytest.mark.parametrize("records", [-1, 0, 1, "two"])
@pytest.mark.parametrize("batch", [False, True])
def test_tiles_of_more_records_than_a_chunk(heget_lib, open_cuts, n, records, batch):
    import torch
    H, ctx, c = heget_lib, open_cuts, CHUNK[n]
    N = 2 * c + 1 if records == "two" else c + records
    tile = -(-N // 4) * 4                     # one tile holds them all
    smp = H.sampler_fixed(500.0)
    w, res = weights(H, ctx, n, N, tile, smp, batch)
    ref, ref_res = weights(H, ctx, n, N, 4, smp)
    assert res.n_pass == ref_res.n_pass == N
    np.testing.assert_array_equal(w, ref)
    mom = torch.empty(N, n + 2, 4, dtype=torch.float64, device="cuda")
    amp = torch.empty(N, dtype=torch.float64, device="cuda")
    H.heget_phase_space_ex(ctx, SEED, 0, N, n, smp, momenta=mom)
    H.heget_amp2(ctx, n, N, mom, amp, precision=H.HEGET_FP64)
    ratio = w / amp.cpu().numpy()             # constant at a fixed energy
    # the generator's momenta rounded to GeV, of any conditioning (no cuts): its typical size, not its tail
    assert np.median(np.abs(ratio / np.median(ratio) - 1)) < 1e-11


@pytest.mark.parametrize("smp", ["toy", "fixed"])
def test_the_default_tile_of_small_calls(heget_lib, gpu, smp):
    import torch
    H, n = heget_lib, 8
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    s = H.sampler_toy_pdf() if smp == "toy" else H.sampler_fixed(500.0)
    H.heget_set_algorithm(gpu, H.HEGET_ALG_SUBSET)
    try:
        ref, _ = weights(H, gpu, n, 32 * sms, 4, s)
        for N in (1, 8, 9, 500, 32 * sms - 1, 32 * sms):
            w, res = weights(H, gpu, n, N, 0, s)
            np.testing.assert_array_equal(w, ref[:N])
            assert res.n_pass == np.count_nonzero(w) and res.n_total == N
            np.testing.assert_allclose(res.sum_w, w.sum(), rtol=1e-13)   # numpy's pairwise sum
    finally:
        H.heget_set_algorithm(gpu, H.HEGET_ALG_TREE)
