"""Tensor-core stages that generate lambda in the kernel: the FP32 plans'
analysis (three BF16 parts, from 8 channels at Nside 512 and 12 at Nside 256)
against the oracle's separable form on sampled coefficients, at the edges of
its tiles (128 l, 64 ring pairs, 8 / 16 channels) and with m and l cut short;
the table plan of the same size must give the same bits.  Bars: relative L2
per channel, FP32 (1e-5).  The streamed plans' bits against the resident ones
are in test_stream_gpu.py; here their widest operand (32 channels a CTA) and a
second channel group at ragged sizes."""
import numpy as np
import pytest
import torch

import oracle
from paper_2510_01785_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


def rel_err(got, ref):
    num = np.linalg.norm((got - ref).reshape(ref.shape[0], -1), axis=1)
    den = np.linalg.norm(ref.reshape(ref.shape[0], -1), axis=1)
    return float(np.max(num / np.maximum(den, 1e-300)))


def sample_lm(lmax, mmax, seed):
    r = syn.rng(seed)
    ls, mm = [], []
    for m in sorted({0, 1, mmax // 3, mmax // 2, mmax - 1 if mmax else 0, mmax}):
        cand = {m, min(m + 1, lmax), min(m + 127, lmax), min(m + 128, lmax), lmax} | set(
            int(x) for x in r.integers(m, lmax + 1, 6))
        ls += sorted(cand)
        mm += [m] * len(cand)
    return np.array(ls, np.int32), np.array(mm, np.int32)


FP32_CASES = [(256, 767, 767, 12), (256, 520, 301, 16), (256, 128, 127, 17), (512, 40, 3, 8), (512, 900, 60, 9)]


@pytest.mark.parametrize("case", FP32_CASES, ids=[f"ns{c[0]}-l{c[1]}-m{c[2]}-b{c[3]}" for c in FP32_CASES])
def test_fp32_analysis_against_oracle(case):
    import paper_2510_01785_gb300 as hpx
    nside, lmax, mmax, nb = case
    maps = syn.white_maps(700 + nside + nb, nside, nb).astype(np.float32)
    x = torch.from_numpy(maps).cuda()
    with hpx.Plan(nside, lmax, mmax, nb, "f32") as p, \
            hpx.Plan(nside, lmax, mmax, nb, "f32", lambda_table=True) as pt:
        a, at = p.map2alm(x), pt.map2alm(x)
        y = p.alm2map_adjoint(x)
        p.device_status()
        assert torch.equal(a, at)
    w = 4 * np.pi / (12 * nside * nside)
    assert rel_err(y.cpu().numpy() * w, a.cpu().numpy()) <= 1e-5
    ls, mm = sample_lm(lmax, mmax, 900 + nside)
    ref = oracle.analysis_sep(maps.astype(np.float64), lmax, ls, mm, weights="equal")
    got = a.cpu().numpy()[:, [m * (2 * lmax + 1 - m) // 2 + l for l, m in zip(ls, mm)]]
    assert rel_err(got, ref) <= 1e-5


@pytest.mark.parametrize("case", [(64, 191, 190, 32), (64, 150, 77, 33), (128, 257, 257, 17)],
                         ids=["ns64-b32", "ns64-b33", "ns128-b17"])
def test_streamed_wide_operands_equal_resident(case):
    import paper_2510_01785_gb300 as hpx
    nside, lmax, mmax, nb = case
    maps = torch.from_numpy(syn.white_maps(60 + nb, nside, nb).astype(np.float32)).cuda()
    alm = torch.from_numpy(syn.gaussian_alm(61 + nb, lmax, mmax, nb).astype(np.complex64)).cuda()
    with hpx.Plan(nside, lmax, mmax, nb, "f32", lambda_table=True, tensor_cores=True) as pr, \
            hpx.Plan(nside, lmax, mmax, nb, "f32", streamed=True) as ps:
        for n in (1, nb // 2, nb):
            ar, as_ = pr.empty_alm(), ps.empty_alm()
            mr, ms = pr.empty_map(), ps.empty_map()
            pr.map2alm_n(n, maps, ar)
            ps.map2alm_n(n, maps, as_)
            pr.alm2map_n(n, alm, mr)
            ps.alm2map_n(n, alm, ms)
            torch.cuda.synchronize()
            assert torch.equal(ar[:n], as_[:n]) and torch.equal(mr[:n], ms[:n]), n
        ps.device_status()


@pytest.mark.parametrize("kind", ["streamed", "fp32"])
def test_expired_wait_is_reported(kind):
    """The copies of the operands withheld (as in test_bounded_wait_gpu.py):
    every CTA's first wait runs out with nothing in flight, the plan reports
    it, and then works as before."""
    import paper_2510_01785_gb300 as hpx
    from paper_2510_01785_gb300 import _lib
    nside, lmax, nb, kw = (64, 191, 4, dict(streamed=True)) if kind == "streamed" else (256, 60, 12, {})
    maps = torch.from_numpy(syn.white_maps(80, nside, nb).astype(np.float32)).cuda()
    alm = torch.from_numpy(syn.gaussian_alm(81, lmax, lmax, nb).astype(np.complex64)).cuda()
    with hpx.Plan(nside, lmax, lmax, nb, "f32", **kw) as p:
        ref_a, ref_m = p.map2alm(maps), p.alm2map(alm)
        p.device_status()
        calls = [lambda: p.map2alm(maps)] + ([lambda: p.alm2map(alm)] if kind == "streamed" else [])
        for call in calls:
            _lib.check(_lib.lib().hpx_plan_test_withhold_copies(p._h, 1), "withhold")
            call()
            with pytest.raises(_lib.HpxError) as e:
                p.device_status()
            assert e.value.status == 4  # HPX_ERR_TIMEOUT
            _lib.check(_lib.lib().hpx_plan_test_withhold_copies(p._h, 0), "withhold")
        assert torch.equal(p.map2alm(maps), ref_a) and torch.equal(p.alm2map(alm), ref_m)
        p.device_status()
