"""FP32 CUDA-core synthesis at the launch widths and splits that
test_f32_channel_counts_gpu.py does not meet: width 4, and three launches (33
channels in widths of 11, 48 in 16).  Each channel as the one-channel plan gives it.
Bar: relative L2 <= 1e-5, the FP32 transforms'."""
import numpy as np
import pytest
import torch

from paper_2510_01785_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb", [4, 33, 48])
@pytest.mark.parametrize("table", [False, True])
def test_channels_alone(nb, table):
    import paper_2510_01785_gb300 as hpx
    nside, lmax = 64, 90
    a = torch.from_numpy(syn.gaussian_alm(690 + nb, lmax, lmax, nb).astype(np.complex64)).cuda()
    with hpx.Plan(nside, lmax, lmax, nb, "f32", lambda_table=table) as p:
        mp = p.alm2map(a)
    with hpx.Plan(nside, lmax, lmax, 1, "f32", lambda_table=table) as p:
        for c in range(nb):
            ref = p.alm2map(a[c: c + 1].clone())[0]
            assert float((mp[c] - ref).double().norm() / ref.double().norm()) <= 1e-5
