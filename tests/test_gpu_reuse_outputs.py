"""fmm_eval_strengths after a full evaluation that wanted fewer outputs (marked
gpu): it allocates nothing, so it can be captured in the default mode, and gives
the bits of a full evaluation with both outputs."""
import pytest

import workloads
from gpu_common import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("batch", [False, True])
def test_stretching_after_a_velocity_only_evaluation(batch):
    import numpy as np
    import torch
    from paper_1106_5273_gb300 import Params, Plan, binding
    n = 3000
    w = workloads.plummer(n)
    pos, gam, sig = to_dev(w["pos"]), to_dev(w["gamma"]), float(workloads.plummer_sigma(n))
    off, sp = np.array([0, 1000, n], np.int64), np.full(2, sig, np.float32)
    vel, dg = torch.zeros((n, 3), device="cuda"), torch.zeros((n, 3), device="cuda")
    prm = Params.default(p=6, theta=0.5, ncrit=32)
    ref, plan = Plan(n, prm), Plan(n, prm)
    if batch:
        want = ref.eval_batch(off, pos, gam, sigma_prob=sp)
        assert binding.lib.fmm_eval_batch(plan._h, 2, off.ctypes.data, pos.data_ptr(), gam.data_ptr(), None,
                                          sp.ctypes.data, None, vel.data_ptr(), None,
                                          torch.cuda.current_stream().cuda_stream) == 0
    else:
        want = ref.eval(pos, gam, sigma_uniform=sig)
        plan.eval(pos, gam, sigma_uniform=sig, vel=vel, stretching=False)
    torch.cuda.synchronize()
    assert torch.equal(vel, want[0])
    held = plan.device_bytes()
    vel.zero_()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, capture_error_mode="global"):
        plan.eval_strengths(gam, vel, dg)
    assert plan.device_bytes() == held
    graph.replay()
    torch.cuda.synchronize()
    assert plan.status() == 0
    assert torch.equal(vel, want[0]) and torch.equal(dg, want[1])
