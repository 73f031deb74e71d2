"""FP32 analyses by the rule that picks the CUDA-core kernel or the tiles that generate
lambda (by channels of the call, lmax and mmax): on either side of each line, n channels
of a wider plan and whole plans give the FP64 plan's coefficients at the FP32 bar
(relative L2 per channel <= 1e-5), the table plan's bits are the recomputing plan's, and
the channels of a call are its own (the rest of the output stays).  Few m or few
channels must not cost more than many."""
import numpy as np
import pytest
import torch

from paper_2510_01785_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nside,lmax,mmax,nb,calls", [
    (256, 300, 120, 17, (1, 8, 9, 16, 17)),  # the channel line at 9, a second group at 17
    (256, 40, 5, 12, (8, 9, 12)),
    (512, 256, 48, 20, (9, 16, 17, 20)),     # 49 m: two launches' worth 98, three 147
    (512, 255, 255, 12, (12,)),              # lmax line
    (512, 256, 98, 9, (4, 5, 8, 9)),         # 99 m
    (512, 256, 99, 9, (4, 5, 8, 9)),         # 100 m
    (1024, 300, 120, 8, (2, 3, 8)),
    (2048, 270, 110, 4, (2, 3, 4)),
])
def test_either_side_of_the_lines(nside, lmax, mmax, nb, calls):
    import paper_2510_01785_gb300 as hpx
    x = torch.from_numpy(syn.white_maps(510 + nside + nb, nside, nb).astype(np.float32)).cuda()
    with hpx.Plan(nside, lmax, mmax, nb, "f64") as p:
        ref = p.map2alm(x.double())
    with hpx.Plan(nside, lmax, mmax, nb, "f32") as p, hpx.Plan(nside, lmax, mmax, nb, "f32", lambda_table=True) as pt:
        for n in calls:
            a, at = p.empty_alm().fill_(7.0), pt.empty_alm()
            p.map2alm_n(n, x, a)
            pt.map2alm_n(n, x, at)
            p.device_status()
            assert torch.equal(a[:n], at[:n]) and bool((a[n:] == 7.0).all())
            err = (a[:n] - ref[:n]).abs().pow(2).sum(1).sqrt() / ref[:n].abs().pow(2).sum(1).sqrt()
            assert float(err.max()) <= 1e-5, (n, err.tolist())


def _best_ms(f):
    for _ in range(3):
        f()
    ms = []
    for _ in range(9):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        f()
        b.record()
        b.synchronize()
        ms.append(a.elapsed_time(b))
    return min(ms)


def test_few_channels_and_few_m_cost_less():
    """One channel of a 16-channel plan is cheaper than a plan of its own plus the
    same again (it took 2.5 times as long as that plan when the plan's channels chose the
    kernel), and 11 of 3072 m cost less than half of 76 (as long, when a CTA took a whole m)."""
    import paper_2510_01785_gb300 as hpx
    x = torch.randn(16, 12 * 256 * 256, device="cuda")
    with hpx.Plan(256, 767, 767, 16, "f32") as p, hpx.Plan(256, 767, 767, 1, "f32") as p1:
        a = p.empty_alm()
        assert _best_ms(lambda: p.map2alm_n(1, x, a)) <= 2.0 * _best_ms(lambda: p1.map2alm_n(1, x, a[:1]))
    x = torch.randn(4, 12 * 2048 * 2048, device="cuda")
    t = []
    for mmax in (10, 75):
        with hpx.Plan(2048, 6143, mmax, 4, "f32") as p:
            a = p.empty_alm()
            t.append(_best_ms(lambda: p.map2alm_n(4, x, a)))
    assert t[0] <= 0.5 * t[1], t
