"""FP64 Legendre stages at every width a launch can have (1 to 8 channels) and
with several launches of equal width: each channel as the one-channel plan gives
it, on one CTA per m and on clusters, with and without the lambda table.
Bar: relative L2 <= 1e-12, the FP64 transforms'."""
import pytest
import torch

from paper_2510_01785_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb", [2, 3, 4, 5, 6, 7, 8, 9, 13, 17])
@pytest.mark.parametrize("nside,lmax,table", [(16, 40, False), (256, 70, False), (16, 47, True)])
def test_channels_alone(nside, lmax, table, nb):
    import paper_2510_01785_gb300 as hpx
    x = torch.from_numpy(syn.white_maps(600 + nb, nside, nb)).cuda()
    a = torch.from_numpy(syn.gaussian_alm(640 + nb, lmax, lmax, nb)).cuda()
    with hpx.Plan(nside, lmax, lmax, nb, "f64", lambda_table=table) as p:
        al, mp = p.map2alm(x), p.alm2map(a)
    with hpx.Plan(nside, lmax, lmax, 1, "f64", lambda_table=table) as p:
        for c in range(nb):
            for got, ref in ((al[c], p.map2alm(x[c: c + 1])[0]), (mp[c], p.alm2map(a[c: c + 1])[0])):
                assert float((got - ref).abs().norm() / ref.abs().norm()) <= 1e-12
