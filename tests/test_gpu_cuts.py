"""The photon cuts' decisions against the oracle's for cuts other than the
default ones: wide and narrow Delta R (beyond pi/3, where the Taylor bounds of
the close pairs stop holding, and beyond pi, where no azimuth separates a
pair), tight and open rapidity windows, no pT cut to speak of."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 3, 4, 5, 8])
@pytest.mark.parametrize("pt,eta,dr", [(20.0, 2.5, 0.4), (20.0, 2.5, 0.01), (5.0, 4.0, 1.2), (5.0, 6.0, 2.0),
                                       (1.0, 6.0, 2.8), (1.0, 8.0, 4.0), (50.0, 0.7, 0.0), (0.0, 12.0, 0.6)])
def test_cut_decisions_match_the_oracle(oracle, heget_lib, gpu, n, pt, eta, dr):
    import torch
    H, N, seed = heget_lib, 4000, 0x0908440300000055
    H.heget_set_params(gpu, pt_min=pt, eta_max=eta, dr_min=dr)
    try:
        for smp, osmp in ((H.sampler_toy_pdf(), oracle.toy_pdf()), (H.sampler_fixed(300.0), oracle.fixed(300.0))):
            mask = torch.empty(N, dtype=torch.uint8, device="cuda")
            H.heget_phase_space_ex(gpu, seed, 17, N, n, smp, mask=mask)
            ref = oracle.phase_space(n, seed, 17, N, osmp, oracle.cuts(pt, eta, dr))["mask"]
            np.testing.assert_array_equal(mask.cpu().numpy().astype(bool), np.asarray(ref).astype(bool))
    finally:
        H.heget_set_params(gpu)


@pytest.mark.parametrize("rs,pt,eta,dr", [(1e-6, 1e-8, 2.5, 0.4), (1e30, 1e28, 2.5, 0.4), (1e60, 1e58, 3.0, 0.4),
                                          (0.02, 1e-9, 30.0, 0.4), (500.0, 0.0, 60.0, 30.0), (500.0, 1e13, 2.5, 0.4),
                                          (9e7, 1e3, 39.0, 0.2)])
def test_cut_decisions_at_the_ends_of_the_fp32_range(oracle, heget_lib, gpu, rs, pt, eta, dr):
    """Events and cuts that FP32 does not hold are decided in FP64."""
    import torch
    H, N, n, seed = heget_lib, 2000, 4, 0x0908440300000056
    H.heget_set_params(gpu, pt_min=pt, eta_max=eta, dr_min=dr)
    try:
        mask = torch.empty(N, dtype=torch.uint8, device="cuda")
        H.heget_phase_space_ex(gpu, seed, 0, N, n, H.sampler_fixed(rs), mask=mask)
        ref = oracle.phase_space(n, seed, 0, N, oracle.fixed(rs), oracle.cuts(pt, eta, dr))["mask"]
        np.testing.assert_array_equal(mask.cpu().numpy().astype(bool), np.asarray(ref).astype(bool))
    finally:
        H.heget_set_params(gpu)
