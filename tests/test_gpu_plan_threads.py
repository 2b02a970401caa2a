"""Plans of different orders on different host threads (marked gpu): each
evaluation gives the bits that its plan gives alone.  The kernels' dynamic
shared memory grows with the order, so no plan may lower another's limit."""
import threading

import pytest

import workloads
from gpu_common import to_dev

pytestmark = pytest.mark.gpu


def test_orders_do_not_disturb_each_other():
    import __graft_entry__
    __graft_entry__.build()
    import torch
    from paper_1106_5273_gb300 import Params, Plan
    n = 3000
    w = workloads.plummer(n)
    pos, gam, sig = to_dev(w["pos"]), to_dev(w["gamma"]), float(workloads.plummer_sigma(n))
    orders = (14, 15, 16, 14, 15, 16)  # 51 to 67 KB for the leaf expansions
    plans = [Plan(n, Params.default(p=p, theta=0.5, ncrit=64)) for p in orders]
    want = [q.eval(pos, gam, sigma_uniform=sig)[0] for q in plans]
    torch.cuda.synchronize()
    errors = []

    def loop(plan, ref):
        try:
            stream = torch.cuda.Stream()
            with torch.cuda.stream(stream):
                for _ in range(150):
                    u, _ = plan.eval(pos, gam, sigma_uniform=sig, stream=stream)
                    stream.synchronize()
                    assert torch.equal(u, ref)
        except Exception as e:  # reported by the test's thread
            errors.append(repr(e))

    threads = [threading.Thread(target=loop, args=a) for a in zip(plans, want)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[:3]
