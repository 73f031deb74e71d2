"""A wide FP32 plan where the device has no room for the operand of its tensor-core
analysis: it is made all the same, without that operand, and its analyses run on
the CUDA cores (relative L2 per channel <= 1e-5 of the other plan's, the FP32 bar)."""
import numpy as np
import pytest
import torch

from paper_2510_01785_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


def test_plan_fits_where_its_operand_does_not():
    import paper_2510_01785_gb300 as hpx
    nside, lmax, mmax, nb = 512, 1535, 1535, 8
    operand = 24 * (mmax + 1) * 2 * nside * nb
    x = torch.from_numpy(syn.white_maps(77, nside, nb).astype(np.float32)).cuda()
    with hpx.Plan(nside, lmax, mmax, nb, "f32") as p:
        ref, held = p.map2alm(x), p.device_bytes
    assert held > operand
    out = torch.empty_like(ref)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    block = torch.empty(free - (held - operand // 2), dtype=torch.uint8, device="cuda")  # half the operand too much
    try:
        with hpx.Plan(nside, lmax, mmax, nb, "f32") as p:
            assert held - p.device_bytes >= operand
            p.map2alm(x, out=out)
            p.device_status()
    finally:
        del block
        torch.cuda.empty_cache()
    err = (out - ref).abs().pow(2).sum(1).sqrt() / ref.abs().pow(2).sum(1).sqrt()
    assert float(err.max()) <= 1e-5
