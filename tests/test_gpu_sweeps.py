"""The upward and downward sweeps at the edges of their splits (marked gpu):
leaves around 8, 16, 32 and 64 particles (8, 4, 2 and 1 thread groups share a
leaf's columns from p = 8 on) against the FP64 oracle FMM, rel-L2 2e-5 (u) and 5e-5 (s) on
the same tree and lists, the allowances of the parity tests; and levels of more
than 1024 cells (four cells per CTA) against levels of few (one), bit by bit:
a problem alone and among its copies in a batch."""
import numpy as np
import pytest

import workloads
from gpu_common import rel_l2, run_fmm, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("p", [3, 8, 9])
@pytest.mark.parametrize("ncrit", [7, 8, 9, 16, 17, 32, 33, 64, 65, 150])
def test_leaf_groups_match_the_oracle(p, ncrit):
    from oracle import fmm as ofmm
    w = workloads.plummer(1200)
    plan, u, s = run_fmm(w, p, 0.4, ncrit, m2l_mode=1)
    ref = ofmm.fmm(w["pos"], w["gamma"], float(w["sigma"]), p, 0.4, ncrit)
    assert rel_l2(u, ref.u) < 2e-5 and rel_l2(s, ref.s) < 5e-5
    plan.close()


@pytest.mark.parametrize("p", [4, 10, 12, 16])
def test_wide_levels_match_narrow_ones(p):
    import torch
    from paper_1106_5273_gb300 import Params, Plan
    w = workloads.plummer(900)
    copies = 24
    prm = Params.default(p=p, theta=0.5, ncrit=4)
    out = []
    for k in (1, copies):
        plan = Plan(900 * k, prm)
        off = np.arange(k + 1, dtype=np.int64) * 900
        u, s = plan.eval_batch(off, to_dev(np.tile(w["pos"], (k, 1))), to_dev(np.tile(w["gamma"], (k, 1))),
                               sigma_prob=np.full(k, w["sigma"], np.float32))
        torch.cuda.synchronize()
        c = plan.cells()
        out.append((u, s, np.bincount(c["level"]).max()))
        plan.close()
    assert out[0][2] < 1024 < out[1][2]
    for a, b in zip(out[0][:2], out[1][:2]):
        assert torch.isfinite(a).all()
        for k in range(copies):
            assert torch.equal(a, b[900 * k:900 * (k + 1)])
