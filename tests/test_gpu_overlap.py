"""With phase timing on, the near and the far field run one after the other on the
caller's stream, otherwise beside each other on two (marked gpu): the same bits
either way, for full, batched and strength-only evaluations."""
import pytest

import workloads
from gpu_common import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("case", ["plummer", "periodic", "widths", "batch", "transpose-simt"])
def test_timing_changes_no_bit(case):
    import __graft_entry__
    __graft_entry__.build()
    import numpy as np
    import torch
    from paper_1106_5273_gb300 import Params, Plan
    kw, sigma = dict(p=8, theta=0.5, ncrit=32), None
    if case == "periodic":
        w = workloads.taylor_green(24)
        kw.update(p=10, theta=0.4, ncrit=64, periodic=1, box_min=w["box_min"], box_len=w["box_len"])
        sig = float(w["sigma"])
    else:
        w = workloads.plummer(20011)
        sig = float(workloads.plummer_sigma(20011))
    n = len(w["pos"])
    if case == "widths":
        sigma = to_dev(sig * np.linspace(0.7, 1.3, n))
    if case == "transpose-simt":
        kw.update(m2l_mode=1, outputs=7)
    pos, gam = to_dev(w["pos"]), to_dev(w["gamma"])
    plan = Plan(n, Params.default(**kw))
    off, sp = np.array([0, 6000, 6001, n]), np.full(3, sig, np.float32)

    def run():
        if case == "batch":
            full = plan.eval_batch(off, pos, gam, sigma_prob=sp)
        else:
            full = plan.eval(pos, gam, sigma=sigma, sigma_uniform=sig)
        again = plan.eval_strengths(gam.flip(0).contiguous())
        torch.cuda.synchronize()
        assert plan.status() == 0
        return full + again

    beside = [run() for _ in range(3)]
    plan.set_timing(True)
    alone = run()
    for other in beside:
        for a, b in zip(alone, other):
            assert torch.equal(a, b)
