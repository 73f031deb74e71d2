"""Streamed plans whose fills go through the two staging buffers: the single-product
and 3xTF32 kinds, and split-product plans of many channels, whose wide analyses are
staged (more than 96 channels of a call from Nside 512, 160 below) while narrower calls
of the same plan, its syntheses and captured calls generate lambda in the kernel.
All give the resident plan's bits; small stages make many blocks."""
import numpy as np
import pytest
import torch

from paper_2510_01785_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


def inputs(nside, lmax, mmax, nb):
    maps = torch.from_numpy(syn.white_maps(820 + nside, nside, 3).astype(np.float32)).cuda()
    alm = torch.from_numpy(syn.gaussian_alm(821 + nside, lmax, mmax, 3).astype(np.complex64)).cuda()
    gain = torch.linspace(0.5, 3.0, nb, device="cuda")[:, None]  # channels of different scales from three fields
    pick = torch.arange(nb, device="cuda") % 3
    return (maps[pick] * gain).contiguous(), (alm[pick] * gain).contiguous()


@pytest.mark.parametrize("dtype", ["f32", "bf16x3"])
@pytest.mark.parametrize("nside,lmax,mmax,nb,stage", [(64, 191, 150, 190, 1 << 20), (128, 200, 40, 161, 0),
                                                      (512, 140, 20, 129, 1 << 20)])
def test_wide_analyses_equal_resident(nside, lmax, mmax, nb, stage, dtype):
    import paper_2510_01785_gb300 as hpx
    maps, alm = inputs(nside, lmax, mmax, nb)
    line = 96 if nside >= 512 else 160
    kw = dict(lambda_table=True, tensor_cores=True) if dtype == "f32" else {}
    with hpx.Plan(nside, lmax, mmax, nb, dtype, **kw) as pr, \
            hpx.Plan(nside, lmax, mmax, nb, dtype, streamed=True, stage_bytes=stage) as ps:
        for n in (1, line, line + 1, nb):
            ar, a = pr.empty_alm(), ps.empty_alm().fill_(7.0)
            pr.map2alm_n(n, maps, ar)
            for _ in range(2):  # the staging buffers alternate
                ps.map2alm_n(n, maps, a)
                torch.cuda.synchronize()
                assert torch.equal(ar[:n], a[:n]) and bool((a[n:] == 7.0).all()), n
        assert torch.equal(pr.alm2map_adjoint(maps), ps.alm2map_adjoint(maps))
        assert torch.equal(pr.alm2map(alm), ps.alm2map(alm))
        ps.device_status()


def test_wide_plan_under_capture():
    import paper_2510_01785_gb300 as hpx
    nside, lmax, nb = 64, 100, 170
    maps, _ = inputs(nside, lmax, lmax, nb)
    with hpx.Plan(nside, lmax, lmax, nb, "f32", streamed=True, stage_bytes=1 << 20) as p:
        ref = p.map2alm(maps).clone()
        x, out = torch.zeros_like(maps), p.empty_alm()
        p.map2alm(x, out=out)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            p.map2alm(x, out=out)
        x.copy_(maps)
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, ref)
        p.device_status()


def test_estimate_bounds_the_wide_plan():
    import paper_2510_01785_gb300 as hpx
    from paper_2510_01785_gb300._lib import lib
    for nside, lmax, nb in ((64, 191, 190), (512, 300, 129)):
        est = lib().hpx_plan_estimate_bytes(nside, lmax, lmax, nb, hpx.DTYPES["f32"], 19)
        with hpx.Plan(nside, lmax, lmax, nb, "f32", streamed=True) as p:
            assert p.device_bytes <= est <= 2 * p.device_bytes, (est, p.device_bytes)


@pytest.mark.parametrize("kind", ["bf16", "tf32x3", "wide"])
def test_staged_analysis_and_synthesis_interleaved(kind):
    """Both stages issued back to back on two streams: the buffers' events keep every
    fill behind the last launch that read its buffer."""
    import paper_2510_01785_gb300 as hpx
    nside, lmax, nb = 64, 191, 170 if kind == "wide" else 4
    dtype, kw, skw = {"bf16": ("bf16", {}, {}), "wide": ("f32", dict(lambda_table=True, tensor_cores=True), {}),
                      "tf32x3": ("f32", dict(lambda_table=True, tensor_cores=True, tf32x3=True), dict(tf32x3=True))}[kind]
    maps, alm = inputs(nside, lmax, lmax, nb)
    with hpx.Plan(nside, lmax, lmax, nb, dtype, **kw) as pr, \
            hpx.Plan(nside, lmax, lmax, nb, dtype, streamed=True, stage_bytes=1 << 20, **skw) as ps:
        ra, rm = pr.map2alm(maps), pr.alm2map(alm)
        torch.cuda.synchronize()
        s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
        outs = [(ps.empty_alm(), ps.empty_map()) for _ in range(4)]
        torch.cuda.synchronize()
        for oa, om in outs:
            with torch.cuda.stream(s1):
                ps.map2alm(maps, out=oa)
            with torch.cuda.stream(s2):
                ps.alm2map(alm, out=om)
        torch.cuda.synchronize()
        for oa, om in outs:
            assert torch.equal(oa, ra) and torch.equal(om, rm)
        ps.device_status()
