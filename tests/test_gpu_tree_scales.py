"""Cell radii of clouds whose squared extents leave the FP32 range at either end
(marked gpu): bit-exact against the oracle at every scale, as the FP64 distances
define them."""
import numpy as np
import pytest

import workloads
from gpu_common import run_fmm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1e-22, 1e-20, 3e-19, 1e-15, 1.0, 1e15, 3e19])
def test_radii_bit_exact_at_any_scale(scale):
    import __graft_entry__
    from oracle import tree as otree
    __graft_entry__.build()
    w = workloads.plummer(5000)
    pos = (w["pos"].astype(np.float64) * scale).astype(np.float32)
    plan, _, _ = run_fmm(dict(pos=pos, gamma=np.zeros_like(pos), sigma=np.float32(scale)), 2, 0.5, 40, m2l_mode=1)
    t = otree.build(pos, 40)[2]
    c = plan.cells()
    assert np.array_equal(c["begin"], t.begin) and np.array_equal(c["center"], t.center)
    assert np.array_equal(c["radius"], t.radius)
