"""Which kernel, form and stream a call takes, checked without a GPU.

tests/host_routes.cu compiles the library's host code (capi.cu) and builds
layout-only plans; every check here is one of its names.
"""
import os
import shutil
import subprocess

import pytest

from paper_2606_13793_gb300 import _build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def host_routes(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    objs = [os.path.join(_build.BUILD_DIR, os.path.splitext(s)[0] + ".o") for s in _build.SOURCES if s != "capi.cu"]
    _build.build(force=not all(os.path.exists(o) for o in objs))
    exe = str(tmp_path_factory.mktemp("host_routes") / "host_routes")
    r = subprocess.run([nvcc, *_build.ARCH, "-O1", "-std=c++17", "--expt-relaxed-constexpr", "-I",
                        os.path.join(ROOT, "include"), "-I", _build.CSRC, os.path.join(ROOT, "tests", "host_routes.cu"),
                        *objs, "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    return exe


CHECKS = ["direct_gemm", "leaf8_streams", "leaf8_batch", "far_order", "near_scratch", "level_kind"]


@pytest.mark.parametrize("check", CHECKS)
def test_route(host_routes, check):
    r = subprocess.run([host_routes, check], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr


def test_shared_memory_limits_are_raised_on_every_device(tmp_path):
    """Kernels of more than 48 KB: the limit is per device (SmemOptIn), and no
    launch sets it in any other way."""
    for name in os.listdir(_build.CSRC):
        text = open(os.path.join(_build.CSRC, name)).read()
        assert text.count("cudaFuncSetAttribute(") == (1 if name == "fmm_internal.h" else 0), name
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path / "host_smem")
    r = subprocess.run([nvcc, *_build.ARCH, "-std=c++17", "-I", _build.CSRC,
                        os.path.join(ROOT, "tests", "host_smem.cu"), "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
