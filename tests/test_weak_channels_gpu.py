"""FP32 analyses of weak channels (small physical units): maps times 2^-105 give
the coefficients times 2^-105 on every path, by channel count (CUDA cores, three
BF16 parts) and beside channels of other magnitudes.  A power of two is exact but for
what falls below the smallest FP32 subnormal: ring values G of rms about 2^-121 lose at
most 2^-150 each, 2^-29 of them.  Bar: relative L2 per channel <= 2^-24."""
import numpy as np
import pytest
import torch

from paper_2510_01785_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nside,lmax,nb,table", [(256, 300, 12, False), (256, 300, 17, True), (256, 300, 4, False),
                                                 (512, 300, 9, False)])
def test_weak_channels(nside, lmax, nb, table):
    import paper_2510_01785_gb300 as hpx
    x = torch.from_numpy(syn.white_maps(330 + nb, nside, nb).astype(np.float32)).cuda()
    scale = torch.ones(nb, 1, device="cuda")
    scale[::2] = 2.0 ** -105
    with hpx.Plan(nside, lmax, lmax, nb, "f32", lambda_table=table) as p:
        for op in ("map2alm", "alm2map_adjoint"):
            ref = getattr(p, op)(x).to(torch.complex128)
            got = getattr(p, op)(x * scale).to(torch.complex128) / scale.double()
            err = (got - ref).abs().pow(2).sum(1).sqrt() / ref.abs().pow(2).sum(1).sqrt()
            assert float(err.max()) <= 2.0 ** -24, (op, err.tolist())
        p.device_status()
