"""A bounded wait that runs out inside an evaluation (marked gpu): the limit is
set so low that the waits give up at once, the evaluation returns FMM_E_TIMEOUT
without using what the waits were for, and the same plan then gives the bits
that it gave before."""
import pytest

import workloads
from gpu_common import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _expires_and_recovers(plan, wait, run):
    import torch
    from paper_1106_5273_gb300 import FmmError
    want = run()
    torch.cuda.synchronize()
    plan.set_wait_limit(wait, -1)
    for _ in range(2):
        with pytest.raises(FmmError) as err:
            run()
        assert err.value.code == -4  # FMM_E_TIMEOUT
        torch.cuda.synchronize()
    plan.set_wait_limit(wait)
    for a, b in zip(run(), want):
        assert torch.equal(a, b)
    plan.close()


@pytest.mark.parametrize("wait", [0, 1, 2])  # octree, traversal, P2P items
@pytest.mark.parametrize("batch", [False, True])
def test_expired_grid_barrier_is_an_error(wait, batch):
    import numpy as np
    from paper_1106_5273_gb300 import Params, Plan
    n = 20000  # about 2000 leaves: every one of the three kernels has several blocks
    w = workloads.plummer(n)
    pos, gam, sig = to_dev(w["pos"]), to_dev(w["gamma"]), float(workloads.plummer_sigma(n))
    plan = Plan(n, Params.default(p=4, theta=0.5, ncrit=16))
    if batch:
        off, sp = np.array([0, 7000, n]), np.full(2, sig, np.float32)
        _expires_and_recovers(plan, wait, lambda: plan.eval_batch(off, pos, gam, sigma_prob=sp))
    else:
        _expires_and_recovers(plan, wait, lambda: plan.eval(pos, gam, sigma_uniform=sig))


@pytest.mark.parametrize("case", ["particles", "particles-batch", "list", "list-batch", "cells", "steps", "buckets"])
def test_expired_look_back_is_an_error(case):
    """A sort waits from its second tile (1024 keys or more) on, so problems of
    at most 1024 particles reach the sorts behind the first."""
    import numpy as np
    from paper_1106_5273_gb300 import Params, Plan
    big = case.startswith(("particles", "list"))
    n = 20000 if big else 1000
    w = workloads.plummer(n)
    pos, gam, sig = to_dev(w["pos"]), to_dev(w["gamma"]), 1e-4
    plan = Plan(n, Params.default(p=4, theta=0.5, ncrit=16 if big else (1 if case == "cells" else 3),
                                  m2l_mode=8 if case == "steps" else 0))
    if case.endswith("batch") or case == "buckets":
        off, sp = np.array([0, 3 * n // 10, n]), np.full(2, sig, np.float32)
        run = lambda: plan.eval_batch(off, pos, gam, sigma_prob=sp)
    else:
        run = lambda: plan.eval(pos, gam, sigma_uniform=sig)
    run()
    st = plan.stats()
    if not big:
        assert (st.ncells > 1024) == (case == "cells")
        assert st.m2l_keys > 1024 and st.m2l_pairs > 1024
    _expires_and_recovers(plan, 4 if case.startswith("list") else 3, run)


def test_bad_limits_are_refused():
    from paper_1106_5273_gb300 import FmmError, Params, Plan
    plan = Plan(8, Params.default())
    for wait, polls in ((-1, 0), (99, 0), (0, (1 << 24) + 1)):
        with pytest.raises(FmmError) as err:
            plan.set_wait_limit(wait, polls)
        assert err.value.code == -1
    plan.close()
