"""The tensor-core M2L at every shape of its two forms (marked gpu): P = p^2
from one coefficient (one MMA of 16 columns) to 256 (one of 256), odd and even
row lengths, one to four K chunks, BF16 and TF32, one problem (work items) and
batches (key buckets), against the FP32 SIMT M2L: rel-L2 1e-5 (u) and 3e-5 (s)
of each other, the tolerance of the parity tests (the FP32 sums set the
difference, not the 2^-18 of the split products)."""
import numpy as np
import pytest

import workloads
from gpu_common import rel_l2, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("mode", [2, 3])
@pytest.mark.parametrize("p", [1, 2, 3, 5, 7, 8, 9, 11, 12, 13, 14, 15, 16])
def test_forms_match_simt(p, mode):
    import torch
    from paper_1106_5273_gb300 import Params, Plan
    w = workloads.plummer(4000)
    w["sigma"] = np.float32(workloads.plummer_sigma(4000))
    pos, gam = to_dev(w["pos"]), to_dev(w["gamma"])
    off = np.array([0, 1500, 4000])
    out = {}
    for m in (1, mode):
        plan = Plan(4000, Params.default(p=p, theta=0.5, ncrit=24, m2l_mode=m))
        u, s = plan.eval(pos, gam, sigma_uniform=float(w["sigma"]))
        ub, sb = plan.eval_batch(off, pos, gam, sigma_prob=np.full(2, w["sigma"], np.float32))
        torch.cuda.synchronize()
        assert plan.stats().m2l_pairs > 0
        out[m] = [a.cpu().numpy() for a in (u, s, ub, sb)]
        plan.close()
    for a, b, tol in zip(out[mode], out[1], (1e-5, 3e-5, 1e-5, 3e-5)):
        assert np.isfinite(a).all() and rel_l2(a, b) < tol
