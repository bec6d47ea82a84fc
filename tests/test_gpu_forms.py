"""The forms one contraction can take, against the oracle and one another.

A small bf16x3 level runs in FP32 in the reflection basis until an M2L schedule
is selected, then on the tensor cores: both forms, the reduced multipole order
and the transposed operator on both, at the precision's parity tolerances (phi
and force 1e-5 for bf16x3, 1e-3 for TF32; adjoint identities the same of
|g| |phi|).  A plan whose variants change between solves (row and
component-major folds, box-major and cell-major densities, folds and bf16
planes, on grids with phantom boxes) gives the bits of a plan built for that
variant: the same kernels on the same values.  The narrow z-run tiles of small
batches give the bits of the wide ones: the same products in the same order.
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import paper_2606_13793_gb300 as fmm  # noqa: E402
from paper_2606_13793_gb300 import _build, inputs  # noqa: E402

TOL = {"bf16x3": 1e-5, "tf32": 1e-3}


@pytest.fixture(scope="module", autouse=True)
def built():
    _build.build()
    assert torch.cuda.is_available()


def rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b))


def plans(shape, p, leaf, prec, **kw):
    """(name, plan) per M2L form: the default and every schedule that exists."""
    plan = fmm.FMMPlan(shape, p, leaf, prec, **kw)
    avail = plan.tc_schedule("m2l")[1]
    yield "default", plan
    plan.close()
    for s in sorted(avail):
        plan = fmm.FMMPlan(shape, p, leaf, prec, **kw)
        try:
            plan.set_tc_schedule("m2l", s)
        except fmm.FMMError:  # no transposed form of that schedule
            plan.close()
            continue
        assert plan.level_kind(plan.leaf_level) == "tensor"
        yield s, plan
        plan.close()


def done(plan, *tensors):
    torch.cuda.synchronize()
    plan.check()
    return [t.double().cpu().numpy() for t in tensors]


@pytest.mark.parametrize("prec", ["bf16x3", "tf32"])
@pytest.mark.parametrize("p,mo", [(4, 3), (6, 5), (6, None)])
def test_small_levels_in_every_form(orc, prec, p, mo):
    rho = inputs.lognormal((64, 48, 80), seed=21).astype(np.float64)
    ref = orc.fmm_orders(rho, 4, p, p if mo is None else mo, p)
    names = []
    for name, plan in plans((64, 48, 80), p, 4, prec, accel=False, mult_order=mo):
        if name == "default":
            assert plan.level_kind(plan.leaf_level) == ("fp32" if prec == "bf16x3" else "tensor")
        (phi,) = done(plan, plan.solve(torch.from_numpy(rho).cuda().float()))
        assert rel(phi, ref) <= TOL[prec], name
        names.append(name)
    assert len(names) >= 2


@pytest.mark.parametrize("prec", ["bf16x3", "tf32"])
def test_transposed_orders_in_every_form(prec):
    rng = np.random.default_rng(8)
    rho, g = (torch.from_numpy(rng.standard_normal((40, 48, 32)).astype(np.float32)).cuda() for _ in range(2))
    names = []
    for name, plan in plans((32, 48, 40), 6, 4, prec, accel=False, mult_order=5):
        phi, grad = plan.solve(rho), plan.solve_adjoint(g)
        done(plan)
        lhs, rhs = float((g.double() * phi.double()).sum()), float((grad.double() * rho.double()).sum())
        scale = float(torch.linalg.vector_norm(g.double()) * torch.linalg.vector_norm(phi.double()))
        assert abs(lhs - rhs) <= TOL[prec] * scale, name
        names.append(name)
    assert len(names) >= 2


def test_analytic_force_in_every_form(orc):
    rho = inputs.lognormal((48, 64, 40), seed=3).astype(np.float64)
    ref = orc.fmm_accel(rho, 4, 6)
    names = []
    for name, plan in plans((48, 64, 40), 6, 4, "bf16x3", accel="analytic"):
        _, acc = done(plan, *plan.solve(torch.from_numpy(rho).cuda().float(), accel=True))
        assert rel(acc, ref) <= TOL["bf16x3"], name
        names.append(name)
    assert len(names) == 3


def test_schedule_selected_between_solves():
    """The reflection form's solve leaves nothing behind that the tensor cores' would read."""
    rho = [torch.rand(52, 28, 36, device="cuda") for _ in range(2)]
    for name, plan in plans((36, 28, 52), 6, 4, "bf16x3", accel=False):
        if name == "default":
            continue
        want = plan.solve(rho[1])
        other = fmm.FMMPlan((36, 28, 52), 6, 4, "bf16x3", accel=False)
        other.solve(rho[0])
        other.set_tc_schedule("m2l", name)
        got = other.solve(rho[1])
        done(other)
        assert torch.equal(got, want), name
        other.close()


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("shape,leaf,kw", [((36, 20, 68), 4, {}), ((18, 34, 26), 2, {}), ((20, 44, 36), 4, {"mult_order": 3}),
                                           ((18, 34, 26), 2, {"final_stage": "m2p"})])
def test_variants_changed_between_solves(prec, shape, leaf, kw):
    variants = [(0, 27), (1, 1), (0, 1), (2, 3), (3, 27), (1, 9), (0, 27), (2, 1), (3, 1)]
    one = fmm.FMMPlan(shape, 5, leaf, prec, **kw)
    # the final-stage M2P takes no variant: its level's is not looked at
    levels = list(range(2, one.leaf_level + (0 if "final_stage" in kw else 1))) + [-1]
    for i, v in enumerate(variants):
        rho = torch.rand(shape[::-1], device="cuda", dtype=one.dtype)
        fresh = fmm.FMMPlan(shape, 5, leaf, prec, **kw)
        for plan in (one, fresh):
            for l in levels:
                plan.set_tuning(l, *v)  # no variant is refused on grids of this size
                assert plan.tuning(l) == v
        got, want = one.solve(rho), fresh.solve(rho)
        got_a, want_a = one.solve_adjoint(rho), fresh.solve_adjoint(rho)
        done(one), done(fresh)
        assert torch.equal(got, want) and torch.equal(got_a, want_a), (i, v)
        fresh.close()
    one.close()


@pytest.mark.parametrize("n,copies", [(192, 7), (256, 6)])
def test_narrow_tiles_give_the_wide_ones_bits(n, copies):
    """The level above the leaf level of one field takes the narrow form (156 + 26
    and 208 + 26 blocks), of several the wide one (from 1216 blocks on)."""
    rho = torch.rand(n, n, n, device="cuda")
    out = []
    for count in (1, copies):
        ps = [fmm.FMMPlan((n,) * 3, 6, 4, "fp32") for _ in range(count)]
        batch = fmm.BatchSolver(ps, autotune=False)
        phis = [torch.empty_like(rho) for _ in ps]
        batch.solve([rho] * count, phis)
        torch.cuda.synchronize()
        assert batch.fused == 1
        out += phis
        batch.close()
        for p in ps:
            p.check()
            p.close()
    assert all(torch.equal(phi, out[0]) for phi in out)
