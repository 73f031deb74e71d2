"""hpx_map2alm_noalloc on plans whose tables are FP16 pairs recomputes lambda in FP32,
and so keeps what is far below an FP16 pair's range: a map that is zero but for the
first rings has coefficients of high m from lambda values down to 2^-126.  Each m
against the recomputing plan's map2alm at the FP32 bar (relative L2 <= 1e-5), as far
as the reference is above 1e-25 of the map."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2510_01785_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kw", [dict(lambda_table=True, tensor_cores=True), dict(streamed=True)], ids=["table", "streamed"])
def test_high_m_of_a_polar_map(kw):
    import paper_2510_01785_gb300 as hpx
    from paper_2510_01785_gb300._lib import check, lib
    nside, lmax, nb = 64, 191, 2
    maps = np.zeros((nb, 12 * nside * nside), np.float32)
    maps[:, :24] = syn.rng(6).standard_normal((nb, 24))  # rings 1 to 3
    x = torch.from_numpy(maps).cuda()
    with hpx.Plan(nside, lmax, lmax, nb, "f32") as p:
        ref = p.map2alm(x).to(torch.complex128)
    with hpx.Plan(nside, lmax, lmax, nb, "f32", **kw) as p:
        out = p.empty_alm()
        check(lib().hpx_map2alm_noalloc(p._h, ctypes.c_void_p(x.data_ptr()), ctypes.c_void_p(out.data_ptr()), None), "noalloc")
        p.device_status()
        got = out.to(torch.complex128)
    compared = 0
    for m in range(lmax + 1):
        base = m * (2 * lmax + 1 - m) // 2
        a, b = got[:, base + m: base + lmax + 1], ref[:, base + m: base + lmax + 1]
        if float(b.norm()) >= 1e-25:
            compared += 1
            assert float((a - b).norm() / b.norm()) <= 1e-5, m
    assert compared >= 20
