"""heget_ward at n = 5 picks its tile by the row count (32 or 48 rows): every
row has the bits that a small tile gives, around both tiles and around the
counts where the choice changes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", [32, 64])
def test_rows_do_not_depend_on_the_tile(heget_lib, gpu, prec):
    import torch
    H, n = heget_lib, 5
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    counts = [1, 31, 32, 33, 47, 48, 49, 32 * sms, 32 * sms + 1] + ([48 * sms, 48 * sms + 1] if prec == 32 else [])
    N = max(counts)
    mom = torch.empty(N, n + 2, 4, dtype=torch.float64, device="cuda")
    H.heget_phase_space_ex(gpu, 0x0908440300006055, 0, N, n, H.sampler_fixed(500.0), momenta=mom)

    def ward(m, tile):
        out = torch.full((m.shape[0],), -1.0, dtype=torch.float64, device="cuda")
        H.heget_set_tile(gpu, n, prec, 0, tile)
        try:
            H.heget_ward(gpu, n, m.shape[0], m, 2, out, precision=prec)
            H.heget_check(gpu)
        finally:
            H.heget_set_tile(gpu, n, prec, 0, 0)
        return out.cpu().numpy()
    ref = ward(mom, 8)
    for c in counts:
        np.testing.assert_array_equal(ward(mom[:c].contiguous(), 0), ref[:c])
