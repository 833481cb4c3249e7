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
