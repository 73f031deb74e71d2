"""The FP32 plans' recurrence where lmax is far above 3 Nside: next to the pole a
chain takes thousands of steps, and its error must stay that of its values'
rounding.  A map that is zero but for one ring gives a_lm = lambda_lm(ring) G_m, one
chain's values times a constant: each (ring, m) against the FP64 plan, up to that
constant (which carries the ring transform's rounding).  Bar: relative L2 over l <=
3 x 2^-24, a rounding each of the value, of its product with G and of that with P_l
(the double-FP32 step's own error is below 2^-28)."""
import numpy as np
import pytest
import torch

from paper_2510_01785_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu

BAR = 3 * 2.0 ** -24


@pytest.mark.parametrize("table", [False, True])
@pytest.mark.parametrize("nside", [64, 128, 256])
def test_rings_next_to_the_pole(nside, table):
    import paper_2510_01785_gb300 as hpx
    lmax, mmax, nb = 16384, 5, 6
    maps = np.zeros((nb, 12 * nside * nside), np.float32)
    r = syn.rng(40 + nside)
    for c in range(nb):  # ring c: 4 (c + 1) pixels from 2 c (c + 1) on
        maps[c, 2 * c * (c + 1): 2 * (c + 1) * (c + 2)] = r.standard_normal(4 * (c + 1))
    x = torch.from_numpy(maps).cuda()
    with hpx.Plan(nside, lmax, mmax, nb, "f64") as p:
        ref = p.map2alm(x.double())
    with hpx.Plan(nside, lmax, mmax, nb, "f32", lambda_table=table) as p:
        got = p.map2alm(x).to(torch.complex128)
        p.device_status()
    worst = 0.0
    for c in range(nb):
        for m in range(mmax + 1):
            base = m * (2 * lmax + 1 - m) // 2
            a, b = got[c, base + m: base + lmax + 1], ref[c, base + m: base + lmax + 1]
            s = torch.vdot(b, a) / torch.vdot(b, b)
            worst = max(worst, float((a - s * b).norm() / (s * b).norm()))
    print(nside, table, np.log2(worst))
    assert worst <= BAR
