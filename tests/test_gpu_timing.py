"""Stage times: no two launches of a stage overlap, so the stages of the
caller's stream add up to no more than the solves took, and a stage of the
levels' stream takes no longer than they did.  Event spans on one stream are
disjoint; 1% and 2 us a launch cover the events' resolution."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import paper_2606_13793_gb300 as fmm  # noqa: E402

CALLER = ("p2m", "m2m", "m2l_tc", "near_field", "near_field_tc", "l2l", "leaf_l2p", "fd_accel")


@pytest.mark.parametrize("shape,prec,accel", [((192, 192, 192), "bf16x3", True), ((256, 128, 192), "tf32", True),
                                              ((192, 160, 128), "bf16x3", "analytic"), ((128, 96, 128), "fp32", True)])
def test_stage_times_fit_in_the_solves(shape, prec, accel):
    plan = fmm.FMMPlan(shape, 6, 4, prec, accel=accel)
    rho = torch.rand(shape[2], shape[1], shape[0], device="cuda")
    for _ in range(3):
        ref = plan.solve(rho, accel=True)
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    torch.cuda.synchronize()
    plan.timing(True)
    a.record()
    for _ in range(5):
        out = plan.solve(rho, accel=True)
    b.record()
    torch.cuda.synchronize()
    ms = a.elapsed_time(b)
    st = plan.timing_read()
    plan.timing(False)
    launches = sum(n for _, n in st.values())
    room = 1.01 * ms + 0.002 * launches
    assert all(n % 5 == 0 for _, n in st.values()) and launches > 0
    assert sum(st[k][0] for k in CALLER) <= room, (ms, st)
    assert all(v <= room for v, _ in st.values()), (ms, st)
    # the launches' order on the streams changes no sum
    assert torch.equal(out[0], ref[0]) and torch.equal(out[1], ref[1])
    plan.check()
    plan.close()
