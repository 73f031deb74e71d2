"""FP32 ring transforms (two transforms of length N / 4 a ring, three radices)
against the FP64 plan's, ring by ring: every transform length's radix is met
(powers of two, convolutions of 16 R, 64 R and 256 R points with each R, direct
sums), with lmax below, at and above the rings' lengths so that bins are zero,
single or folded.  Bar: relative L2 of the pixels of each ring and its mirror
(synthesis; E + O and E - O of the same sums, one of which may cancel) and of each
m's coefficients (analysis) <= 1e-5, as for the FP32 transforms."""
import numpy as np
import pytest
import torch

from paper_2510_01785_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu

CASES = [(1, 40, 2), (8, 23, 3), (16, 200, 1), (64, 191, 5), (256, 520, 1), (512, 300, 2), (1024, 150, 1), (2048, 260, 1)]


@pytest.mark.parametrize("case", CASES, ids=[f"ns{c[0]}-l{c[1]}-b{c[2]}" for c in CASES])
def test_rings_against_fp64(case):
    import paper_2510_01785_gb300 as hpx
    nside, lmax, nb = case
    alm = syn.gaussian_alm(900 + nside, lmax, lmax, nb, power=0.0).astype(np.complex64)
    maps = syn.white_maps(950 + nside, nside, nb).astype(np.float32)
    a, x = torch.from_numpy(alm).cuda(), torch.from_numpy(maps).cuda()
    with hpx.Plan(nside, lmax, lmax, nb, "f64") as p:
        m64, a64 = p.alm2map(a.to(torch.complex128)), p.map2alm(x.double())
    with hpx.Plan(nside, lmax, lmax, nb, "f32") as p:
        m32, a32 = p.alm2map(a).double(), p.map2alm(x).to(torch.complex128)
    i = np.concatenate([np.arange(1, nside), np.full(2 * nside + 1, nside), np.arange(nside - 1, 0, -1)])
    y = np.arange(4 * nside - 1)
    ring = torch.from_numpy(np.repeat(np.minimum(y, 4 * nside - 2 - y), 4 * i)).cuda()
    m = torch.from_numpy(np.repeat(np.arange(lmax + 1), np.arange(lmax + 1, 0, -1))).cuda()
    for got, ref, key in ((m32, m64, ring), (a32, a64, m)):
        n = int(key.max()) + 1
        for c in range(nb):
            num = torch.zeros(n, dtype=torch.float64, device="cuda").index_add_(0, key, (got[c] - ref[c]).abs() ** 2)
            den = torch.zeros(n, dtype=torch.float64, device="cuda").index_add_(0, key, ref[c].abs() ** 2)
            assert float((num / den).sqrt().max()) <= 1e-5
