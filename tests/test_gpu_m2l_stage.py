"""The whole-step pipeline stage of the tensor-core M2L (marked gpu) is taken
where two CTAs with such a stage fit an SM: p = 9 and 10, not p = 11, whose
operators fill all 128 rows.  Whatever the stage, the bits are those of one K
chunk per stage, and the SIMT M2L agrees within the parity tests' tolerances."""
import numpy as np
import pytest

import workloads
from gpu_common import rel_l2, run_fmm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,chunks", [(9, 2), (10, 2), (11, 1)])
def test_whole_step_stage_where_two_ctas_fit(p, chunks):
    import __graft_entry__
    __graft_entry__.build()
    from paper_1106_5273_gb300 import FMM_M2L_CHUNK_STAGES
    w = dict(workloads.plummer(4000), sigma=np.float32(workloads.plummer_sigma(4000)))
    plan, u, s = run_fmm(w, p, 0.4, 24, m2l_mode=2)
    assert plan.stats().m2l_pairs > 0 and plan.stats().m2l_stage_chunks == chunks
    _, uc, sc = run_fmm(w, p, 0.4, 24, m2l_mode=2 | FMM_M2L_CHUNK_STAGES)
    assert np.array_equal(u, uc) and np.array_equal(s, sc)
    _, us, ss = run_fmm(w, p, 0.4, 24, m2l_mode=1)
    assert rel_l2(u, us) < 1e-5 and rel_l2(s, ss) < 3e-5


def test_simt_tiles_are_wide_at_every_p():
    """The SIMT M2L takes tiles of 64 cells whatever P is, so the steps are the
    same at every order (the tensor-core M2L takes smaller ones at p = 12)."""
    import __graft_entry__
    __graft_entry__.build()
    w = dict(workloads.plummer(12000), sigma=np.float32(workloads.plummer_sigma(12000)))
    steps = {(p, mode): run_fmm(w, p, 0.5, 16, m2l_mode=mode)[0].stats().m2l_steps
             for p, mode in ((4, 1), (10, 1), (12, 1), (12, 2))}
    assert steps[4, 1] == steps[10, 1] == steps[12, 1] < steps[12, 2]
