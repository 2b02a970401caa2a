"""The frontier loop on both sides of its rule (marked gpu): 4096 leaves of one
blob each and a MAC that accepts nothing, so that the last frontier holds
4096 x 512 pairs (a thread per pair) and the first ones a few (a lane per
child).  Every pair is counted once, and the result is the pair sum: rel-L2
2e-5 (u) and 5e-5 (s) against the FP64 direct sum, FP32 unit roundoff times the
growth of a 4096-term sum (a few hundred)."""
import pytest

import workloads
from gpu_common import rel_l2, run_fmm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tie", [0, 1])
def test_frontier_of_all_pairs(tie):
    import __graft_entry__
    from oracle import direct as od
    __graft_entry__.build()
    w = workloads.jittered_lattice(16)
    n = w["pos"].shape[0]
    plan, u, s = run_fmm(w, 4, 1e-3, 1, split_tie=tie)
    st = plan.stats()
    assert st.nleaves > 4000 and st.m2l_pairs == 0
    assert st.p2p_cell_pairs == st.nleaves ** 2 and st.p2p_pairs == n * n
    ud, sd = od.direct(w["pos"], w["gamma"], w["pos"], w["gamma"], float(w["sigma"]), skip_self=True)
    assert rel_l2(u, ud) < 2e-5 and rel_l2(s, sd) < 5e-5
    plan.close()
