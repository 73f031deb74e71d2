"""Slots of small maps overtake the kernels of large ones: while a large slot has
syntheses queued, a small batch of both operations must be through in half the time of
one of them (on streams of equal priority it took longer than one).  Results stay those of the transforms alone, and a call gives the
same bits on streams of any priority (from Nside 512 the ring stages fork on default
streams only)."""
import numpy as np
import pytest
import torch

from paper_2510_01785_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


def test_small_batches_overtake_large_ones():
    from paper_2510_01785_gb300.serve import GpuExecutor, Request
    ex = GpuExecutor(keep_outputs=False, lambda_table_nsides=(64,), batch_channels={64: 8, 1024: 32}, streamed_nsides=(1024,))
    big, small = ex.new_slot(1024, 3071, 32), ex.new_slot(64, 191, 8)
    try:
        rb = Request(0, "alm2map", 1024, 32, x=torch.view_as_complex(torch.randn(32, big["plan"].nalm, 2, device="cuda")))
        rs = Request(1, "alm2map", 64, 8, x=torch.view_as_complex(torch.randn(8, small["plan"].nalm, 2, device="cuda")))
        ra = Request(2, "map2alm", 64, 8, x=torch.randn(8, small["plan"].npix, device="cuda"))

        def timed(slot, calls):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record(slot["stream"])
            for op, r in calls:
                ex.launch(slot, op, [r])
            b.record(slot["stream"])
            return a, b
        pair = [("alm2map", rs), ("map2alm", ra)]
        timed(big, [("alm2map", rb)])
        timed(small, pair)
        torch.cuda.synchronize()
        b0, b1 = timed(big, [("alm2map", rb)] * 8)
        s0, s1 = timed(small, pair)
        torch.cuda.synchronize()
        assert s0.elapsed_time(s1) <= 0.5 * b0.elapsed_time(b1) / 8, (s0.elapsed_time(s1), b0.elapsed_time(b1))
    finally:
        ex.free_slot(big)
        ex.free_slot(small)


def test_same_bits_on_streams_of_any_priority():
    import paper_2510_01785_gb300 as hpx
    nside, lmax, nb = 512, 200, 3
    maps = torch.from_numpy(syn.white_maps(31, nside, nb).astype(np.float32)).cuda()
    alm = torch.from_numpy(syn.gaussian_alm(32, lmax, lmax, nb).astype(np.complex64)).cuda()
    for dtype in ("f32", "bf16", "f64"):
        x, a = (maps.double(), alm.to(torch.complex128)) if dtype == "f64" else (maps, alm)
        with hpx.Plan(nside, lmax, lmax, nb, dtype) as p:
            ra, rm = p.map2alm(x).clone(), p.alm2map(a).clone()
            torch.cuda.synchronize()
            for prio in (-1, -3):
                s = torch.cuda.Stream(priority=prio)
                with torch.cuda.stream(s):
                    ga, gm = p.map2alm(x), p.alm2map(a)
                s.synchronize()
                assert torch.equal(ga, ra) and torch.equal(gm, rm)
