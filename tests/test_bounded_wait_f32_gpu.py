"""The bounded waits of the FP32 analysis on the CUDA cores, made to run out on
purpose without a fault (as in test_bounded_wait_gpu.py): the compute warps withhold
their blocks' sums, so every CTA's summing warp gives up after 1 s and sends nothing,
and every output warp does.  The plan must report HPX_ERR_TIMEOUT and give the same
bits as before once the sums flow again.  One CTA a cluster (Nside 64) and several
(Nside 256, 512), more blocks of l than the inbox has places, every CTA resident."""
import numpy as np
import pytest
import torch

from paper_2510_01785_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nside,lmax,mmax,nb,table", [(64, 191, 10, 3, False), (256, 400, 10, 8, False),
                                                      (256, 300, 4, 2, True), (512, 200, 10, 1, False)])
def test_withheld_sums_time_out_and_the_plan_recovers(nside, lmax, mmax, nb, table):
    import paper_2510_01785_gb300 as hpx
    from paper_2510_01785_gb300._lib import HpxError, check, lib
    maps = torch.from_numpy(syn.white_maps(440 + nside, nside, nb).astype(np.float32)).cuda()
    with hpx.Plan(nside, lmax, mmax, nb, "f32", lambda_table=table) as p:
        ref = p.map2alm(maps).clone()
        p.device_status()
        check(lib().hpx_plan_test_withhold_copies(p._h, 1), "withhold")
        p.map2alm(maps)
        with pytest.raises(HpxError) as err:
            p.device_status()
        assert err.value.status == 4  # HPX_ERR_TIMEOUT
        check(lib().hpx_plan_test_withhold_copies(p._h, 0), "withhold")
        p.device_status()  # the record was cleared
        assert torch.equal(p.map2alm(maps), ref)
        p.device_status()
