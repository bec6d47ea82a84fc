"""Reflection-basis contractions (csrc/k_sym.cu).

CPU: the weight tables of both forms, contracted as the kernels contract them,
equal the direct contraction with the plan's weight functions (every order,
reduced multipole or local orders, the near field) to 1e-13 of the terms.

GPU: grids at the edges of the tiles (8 x 4 x 8 / 4 / 2 rows, 32- and 8-row
chunks): extents of one box past a tile, flat and elongated grids, the
smallest tree; every variant, against the FP64 oracle at the parity
tolerances of the direct form (rounding of the same sums: FP64 1e-10, FP32
1e-5), and the adjoint of a reduced multipole order by <g, A r> = <A^T g, r>.
"""
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_2606_13793_gb300 import _build, inputs

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
TOL = {"fp64": 1e-10, "fp32": 1e-5}


def test_reflection_weights_equal_the_direct_contraction(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    objs = [os.path.join(_build.BUILD_DIR, os.path.splitext(s)[0] + ".o") for s in _build.SOURCES if s != "capi.cu"]
    _build.build(force=not all(os.path.exists(o) for o in objs))
    exe = str(tmp_path / "host_reflection")
    src = os.path.join(ROOT, "tests", "host_reflection.cu")
    r = subprocess.run([nvcc, *_build.ARCH, "-O1", "-std=c++17", "--expt-relaxed-constexpr", "-I",
                        os.path.join(ROOT, "include"), "-I", _build.CSRC, src, *objs, "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    print(r.stdout)
    assert r.returncode == 0, r.stdout + r.stderr
    assert r.stdout.count("reflection m2l") == 12 and r.stdout.count("reflection M2P") == 3


def _rel(a, b):
    return float(np.linalg.norm(np.asarray(a, np.float64) - b) / np.linalg.norm(b))


def _solve(plan, rho):
    import torch

    phi = plan.solve(torch.from_numpy(rho).cuda().to(plan.dtype))
    torch.cuda.synchronize()
    plan.check()
    return phi.double().cpu().numpy()


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("shape,p", [((16, 16, 16), 6), ((36, 20, 68), 5), ((72, 36, 20), 8), ((8, 64, 132), 7),
                                     ((132, 68, 36), 2)])
def test_reflection_forms_match_oracle(orc, prec, shape, p):
    import paper_2606_13793_gb300 as fmm

    if prec == "fp64" and p == 8:
        p = 7  # FP64 order 8 keeps the Cartesian M2L
    rho = inputs.plummer(shape, seed=p).astype(np.float64)
    ref = orc.fmm(rho, 4, p)["phi"]
    for variant in (None, (0, 27), (0, 1), (3, 27), (3, 1), (1, 1), (1, 9), (2, 3), (2, 1)):
        plan = fmm.FMMPlan(shape, p, 4, prec)
        if variant:
            for lvl in list(range(2, plan.leaf_level + 1)) + [-1]:
                try:
                    plan.set_tuning(lvl, *variant)
                except fmm.FMMError:
                    pass  # the split scratch does not hold this variant
        err = _rel(_solve(plan, rho), ref)
        assert err <= TOL[prec], (variant, err)
        plan.close()


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("shape,p,leaf,mo", [((16, 16, 16), 3, 2, 2), ((18, 34, 66), 4, 2, None),
                                             ((36, 20, 68), 4, 4, 3), ((130, 10, 22), 2, 2, None)])
def test_reflection_m2p_and_leaf2_near_field_match_oracle(orc, prec, shape, p, leaf, mo):
    import paper_2606_13793_gb300 as fmm

    rho = inputs.plummer(shape, seed=p).astype(np.float64)
    ref = orc.fmm_orders(rho, leaf, p, p if mo is None else mo, p, "m2p")
    for near in (None, (1, 1), (2, 3), (0, 1)):
        plan = fmm.FMMPlan(shape, p, leaf, prec, final_stage="m2p", mult_order=mo)
        if near:
            try:
                plan.set_tuning(-1, *near)
            except fmm.FMMError:
                pass  # the split scratch does not hold this variant
        err = _rel(_solve(plan, rho), ref)
        assert err <= TOL[prec], (near, err)
        plan.close()


@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(36, 24, 44), (64, 64, 64)])
def test_reflection_adjoint_of_reduced_multipole_order(shape):
    import torch

    import paper_2606_13793_gb300 as fmm

    plan = fmm.FMMPlan(shape, 5, 4, "fp64", accel=False, mult_order=3)
    g = torch.Generator(device="cuda").manual_seed(5)
    s = (shape[2], shape[1], shape[0])
    r = torch.rand(s, device="cuda", dtype=torch.float64, generator=g)
    w = torch.rand(s, device="cuda", dtype=torch.float64, generator=g)
    a = float((w * plan.solve(r)).sum())
    b = float((plan.solve_adjoint(w) * r).sum())
    plan.check()
    assert abs(a - b) <= 1e-12 * abs(a)
    plan.close()
