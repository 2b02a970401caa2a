"""The plan's operator cache (marked gpu): translations are looked up in a
device table, missing ones built once.  Evaluations that hit, extend and miss
the cache give the bits of a fresh plan."""
import numpy as np
import pytest

import workloads
from gpu_common import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("mode", [0, 8])  # steps from bins, steps by sorting
@pytest.mark.parametrize("p", [4, 10])
def test_cached_operators_give_the_same_bits(p, mode):
    import torch
    from paper_1106_5273_gb300 import Params, Plan
    clouds = [workloads.plummer(3000, seed=s) for s in (1, 2)] + [workloads.uniform_ball(2500, seed=3)]
    for w in clouds:
        w["sigma"] = np.float32(0.02)

    def run(plan, w):
        u, s = plan.eval(to_dev(w["pos"]), to_dev(w["gamma"]), sigma_uniform=float(w["sigma"]))
        torch.cuda.synchronize()
        return u.cpu().numpy(), s.cpu().numpy(), plan.stats()

    kept = Plan(3000, Params.default(p=p, theta=0.5, ncrit=16, m2l_mode=mode))
    seen = 0
    for turn in range(2):
        for w in clouds:
            fresh = Plan(3000, Params.default(p=p, theta=0.5, ncrit=16, m2l_mode=mode))
            u0, s0, st0 = run(fresh, w)
            u1, s1, st1 = run(kept, w)
            assert st0.m2l_keys > 0 and st0.m2l_built == st0.m2l_keys == st1.m2l_keys
            assert st1.m2l_built == 0 if turn else st1.m2l_built <= st1.m2l_keys
            seen += st1.m2l_built
            assert np.array_equal(u0, u1) and np.array_equal(s0, s1)
            fresh.close()
    assert seen > 0
    kept.close()
