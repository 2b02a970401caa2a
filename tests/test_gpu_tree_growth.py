"""The cooperative octree kernel stops when a level outgrows the cell arrays
and resumes after they grew (marked gpu): small leaves on a deep cloud need
more cells than the starting capacity; the cells stay bit-exact against the
oracle, also where the coordinates dwarf the cells."""
import numpy as np
import pytest

import workloads
from gpu_common import run_fmm

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("n,ncrit,shift", [(1, 1, 0.0), (2, 1, 0.0), (700, 1, 0.0), (5000, 1, 0.0), (5000, 2, 300.0),
                                           (40000, 3, 0.0), (40000, 4096, -7.0)])
def test_cells_bit_exact_through_growth(n, ncrit, shift):
    from oracle import tree as otree
    w = workloads.plummer(n)
    w["pos"] = (w["pos"] + np.float32(shift)).astype(np.float32)
    w["gamma"][:] = 0.0
    plan, _, _ = run_fmm(dict(w, sigma=np.float32(1e-6)), 2, 0.5, ncrit, m2l_mode=1)
    t = otree.build(w["pos"], ncrit)[2]
    c = plan.cells()
    assert len(c["begin"]) == len(t.begin)
    for f in ("begin", "end", "level", "parent"):
        assert np.array_equal(c[f].astype(np.int64), getattr(t, f)), f
    assert np.array_equal(c["center"], t.center) and np.array_equal(c["radius"], t.radius)
