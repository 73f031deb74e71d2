"""FP32 CUDA-core synthesis at the widths a launch can have (1, 2, 3, 4, 6, 8, 12,
16 channels) and with several launches: each channel as the one-channel plan gives
it, recomputing lambda and from the table.  Bar: relative L2 <= 1e-5, the FP32
transforms'."""
import numpy as np
import pytest
import torch

from paper_2510_01785_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb", [2, 3, 5, 6, 7, 9, 12, 13, 17, 20])
@pytest.mark.parametrize("nside,lmax,table", [(16, 40, False), (128, 200, False), (16, 47, True)])
def test_channels_alone(nside, lmax, table, nb):
    import paper_2510_01785_gb300 as hpx
    a = torch.from_numpy(syn.gaussian_alm(680 + nb, lmax, lmax, nb).astype(np.complex64)).cuda()
    with hpx.Plan(nside, lmax, lmax, nb, "f32", lambda_table=table) as p:
        mp = p.alm2map(a)
    with hpx.Plan(nside, lmax, lmax, 1, "f32", lambda_table=table) as p:
        for c in range(nb):
            ref = p.alm2map(a[c: c + 1].clone())[0]  # (a slice need not be 16-byte aligned)
            assert float((mp[c] - ref).double().norm() / ref.double().norm()) <= 1e-5
