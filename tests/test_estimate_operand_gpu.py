"""hpx_plan_estimate_bytes of plans with operands or tables that its other test does
not meet: the tensor-core analysis of wide FP32 plans (8 and 16 channels a group, one
group and more) and plans on either side of the rule that makes it, and the second
chain starts of small FP16 hi/lo plans.  An upper bound, and not a loose one."""
import pytest

pytestmark = pytest.mark.gpu

CASES = [  # nside, lmax, mmax, nbatch, Plan keywords, flags
    (256, 767, 767, 12, {}, 0),
    (256, 767, 767, 11, {}, 0),
    (256, 767, 400, 33, {}, 0),
    (512, 700, 700, 8, {}, 0),
    (512, 255, 255, 8, {}, 0),
    (512, 300, 200, 9, dict(lambda_table=True), 1),
    (64, 191, 191, 17, dict(lambda_table=True, tensor_cores=True), 3),
]


@pytest.mark.parametrize("case", CASES, ids=[f"ns{c[0]}-l{c[1]}-m{c[2]}-b{c[3]}-flags{c[5]}" for c in CASES])
def test_estimate_bounds_the_plan(case):
    import paper_2510_01785_gb300 as hpx
    from paper_2510_01785_gb300._lib import lib
    nside, lmax, mmax, nb, kw, flags = case
    est = lib().hpx_plan_estimate_bytes(nside, lmax, mmax, nb, hpx.DTYPES["f32"], flags)
    with hpx.Plan(nside, lmax, mmax, nb, "f32", **kw) as p:
        held = p.device_bytes
    assert held <= est <= 2 * held, (held, est)
