"""The products that the benchmark counts for a fused batch are those that the
library's batch tables multiply: the form of every item (reflection basis or
direct) as the tables give it, per leaf size and precision."""
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

import bench  # noqa: E402
from test_routes import host_routes  # noqa: E402,F401  (the fixture)


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("leaf,p,n", [(2, 4, 32), (4, 6, 64), (4, 1, 64), (4, 3, 16), (8, 4, 64), (8, 1, 64)])
def test_batch_products_follow_the_batch_tables(host_routes, fp64, leaf, p, n):  # noqa: F811
    import subprocess

    r = subprocess.run([host_routes, "batch_forms", str(n), str(p), str(leaf), str(int(fp64))], capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
    mirror = [int(v) for v in r.stdout.split()]  # levels 2 .. leaf level, then the near field
    lev = bench.hierarchy((n,) * 3, leaf)
    assert len(mirror) == len(lev) - 1
    want = sum(bench.m2l_flop_level((n,) * 3, leaf, p, l, p >= 2) / (8 if mirror[l - 2] else 1)
               for l in range(2, len(lev)))
    want += bench.algorithmic_counts((n,) * 3, leaf, p)["near_flop"] / (8 if mirror[-1] else 1)
    assert bench.batch_products([n], leaf, p, fp64) == pytest.approx(want, rel=1e-12)
