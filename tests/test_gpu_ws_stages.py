"""The warp-specialised kernels over several stages a block (ring slots,
harvest, the sampler's warp and its hand-over start at a block's third stage),
a ragged last one included, against the FP64 tile kernel, whose threads draw
for themselves: the same cut decisions, counts and attempts, the same weights.
Samplers: the toy PDF as it is, with a floor that most pairs of fractions miss
and few tries (draws that run out), and uniform energies."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SEED = 0x09084403000000D1
STAGE = {2: 128, 3: 128, 4: 128, 5: 64, 6: 64, 7: 96, 8: 64}    # producers of a block


def samplers(H):
    return {"toy": H.sampler_toy_pdf(), "uniform": H.sampler_uniform(500.0, 2000.0),
            "floor1": H.sampler_toy_pdf(floor=2500.0, max_tries=1), "floor2": H.sampler_toy_pdf(floor=9000.0, max_tries=2),
            "floor3": H.sampler_toy_pdf(floor=300.0, max_tries=3)}


def xsec(H, ctx, n, N, smp, prec, seed=SEED):
    import torch
    w = torch.full((N,), -1.0, dtype=torch.float64, device="cuda")
    res = torch.zeros(80, dtype=torch.uint8, device="cuda")
    H.heget_xsec_async(ctx, n, seed, 7, N, smp, prec, res, w_out=w)
    return w.cpu().numpy(), H.result_from_tensor(res)


@pytest.fixture(params=[(2, 0), (3, 0), (4, 0), (5, 0), (3, 1), (4, 1), (6, 1), (7, 1), (8, 1)], ids=lambda p: f"n{p[0]}alg{p[1]}")
def setup(request, heget_lib, gpu):
    n, alg = request.param
    heget_lib.heget_set_algorithm(gpu, alg)
    yield gpu, n
    heget_lib.heget_set_algorithm(gpu, heget_lib.HEGET_ALG_TREE)


@pytest.mark.parametrize("smp", ["toy", "uniform", "floor1", "floor2", "floor3"])
def test_several_stages_a_block(heget_lib, setup, smp):
    import torch
    H, (ctx, n) = heget_lib, setup
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    blocks = sms * (1 if n >= 7 else 3)       # resident blocks, at most
    s = samplers(H)[smp]
    for N in (STAGE[n] * (4 * blocks) + 1, STAGE[n] * (2 * blocks + 1) - 1):
        w32, r32 = xsec(H, ctx, n, N, s, 32)
        w64, r64 = xsec(H, ctx, n, N, s, 64)
        np.testing.assert_array_equal(w32 == 0, w64 == 0)
        assert (r32.n_pass, r32.n_total, r32.n_tries) == (r64.n_pass, r64.n_total, r64.n_tries)
        assert r32.n_pass == np.count_nonzero(w32) and r32.n_total == N
        on = w64 != 0
        if on.any():
            rel = np.abs(w32[on] / w64[on] - 1)
            # the stated FP32 error, and the parity tests' tail
            assert np.median(rel) <= 2e-6 and rel.max() <= 1e-3


@pytest.mark.parametrize("n,alg", [(2, 0), (3, 0), (4, 0), (7, 1)])
@pytest.mark.parametrize("smp", ["floor1", "floor2", "floor3"])
def test_draws_that_run_out_against_the_oracle(oracle, heget_lib, gpu, n, alg, smp):
    H, N = heget_lib, 3000
    s = samplers(H)[smp]
    o = oracle.toy_pdf(floor=s.floor, max_tries=s.max_tries)
    ref = oracle.phase_space(n, SEED, 7, N, o, oracle.cuts())
    assert np.count_nonzero(ref["weight"] == 0) > 0          # some draws run out (floor2: all of them)
    H.heget_set_algorithm(gpu, alg)
    try:
        w, r = xsec(H, gpu, n, N, s, 32)
    finally:
        H.heget_set_algorithm(gpu, H.HEGET_ALG_TREE)
    np.testing.assert_array_equal(w != 0, np.asarray(ref["mask"]).astype(bool))
    assert r.n_pass == np.count_nonzero(ref["mask"]) and r.n_tries == int(ref["tries"].sum())


@pytest.mark.parametrize("n", [2, 3, 4, 5])
def test_kernels_of_the_fp32_tree_give_the_same_bits(heget_lib, gpu, n):
    """The warp-specialised kernel, the tile kernel and the batch kernel."""
    import torch
    H, N, s = heget_lib, 30_011, heget_lib.sampler_toy_pdf()
    ws, _ = xsec(H, gpu, n, N, s, 32)
    H.heget_set_tile(gpu, n, 32, 1, 128)
    try:
        tile, _ = xsec(H, gpu, n, N, s, 32)
    finally:
        H.heget_set_tile(gpu, n, 32, 1, 0)
    w = torch.empty(N, dtype=torch.float64, device="cuda")
    res = torch.zeros(80, dtype=torch.uint8, device="cuda")
    H.heget_xsec_batch(gpu, [dict(n=n, precision=32, seed=SEED, i0=7, N=N, sampler=s, result_dev=res, w_out=w)])
    np.testing.assert_array_equal(tile, ws)
    np.testing.assert_array_equal(w.cpu().numpy(), ws)


@pytest.mark.parametrize("n", [4, 5])
def test_warp_rounds_at_the_stated_errors(oracle, heget_lib, gpu, n):
    """heget_amp2 of events that pass the cuts, both precisions, against the oracle."""
    import torch
    from helpers import fp64_tolerance
    H = heget_lib
    ps = oracle.phase_space(n, SEED + n, 0, 900 if n == 4 else 300, oracle.toy_pdf(), oracle.cuts())
    mom = ps["momenta"][np.asarray(ps["mask"]).astype(bool)]
    ref = oracle.amp2(n, mom)
    out = torch.empty(len(mom), dtype=torch.float64, device="cuda")
    dev = torch.from_numpy(np.ascontiguousarray(mom)).cuda()
    H.heget_amp2(gpu, n, len(mom), dev, out, precision=64)
    assert np.all(np.abs(out.cpu().numpy() / ref - 1) <= fp64_tolerance(mom))
    H.heget_amp2(gpu, n, len(mom), dev, out, precision=32)
    assert np.median(np.abs(out.cpu().numpy() / ref - 1)) <= 2e-6
