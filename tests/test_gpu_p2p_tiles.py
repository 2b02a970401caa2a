"""The pair kernel at the edges of its tiles (marked gpu): leaves of 1 to 130
targets (lane groups of 8, 16 and 32 targets, two targets per lane beyond 32,
several tiles beyond 64), source chunks that span many leaves, lists split
into ranges, zero-strength sources, one core width, one per particle and the
mixed rule.  theta = 1e-3 leaves no M2L pair, so the result is the pair sum:
rel-L2 within 2e-5 (u) and 5e-5 (s) of the FP64 sum -- FP32 unit roundoff
6e-8 times the growth of a 700-term sum in leaf-relative coordinates (at
most a few hundred) -- and every pair is counted once."""
import numpy as np
import pytest

import workloads
from gpu_common import rel_l2, to_dev

pytestmark = pytest.mark.gpu

N = 700


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.fixture(scope="module")
def sums():
    from oracle import pairs
    w = workloads.plummer(N)
    sig0 = np.float32(workloads.plummer_sigma(N))
    sig = (sig0 * np.linspace(0.7, 1.3, N)).astype(np.float32)
    gam = w["gamma"].copy()
    gam[::7] = 0.0  # zero strengths are left out of the staged chunks
    x, g = w["pos"].astype(np.float64), gam.astype(np.float64)
    skip = np.eye(N, dtype=bool)
    out = {}
    for kind, s, st in (("one", np.full(N, float(sig0)), None), ("each", sig.astype(np.float64), None),
                        ("mixed", sig.astype(np.float64), sig.astype(np.float64))):
        for tr in (False, True):
            out[kind, tr] = pairs.pair_sum(x, g, x, g, s, None, skip, transpose=tr, sig_t=st)
    return w["pos"], gam, sig0, sig, out


@pytest.mark.parametrize("kind", ["one", "each", "mixed"])
@pytest.mark.parametrize("ncrit", [1, 8, 9, 16, 17, 32, 33, 64, 65, 130])
def test_pair_sums_at_tile_edges(sums, ncrit, kind):
    import torch
    from paper_1106_5273_gb300 import FMM_SIGMA_MIXED, Params, Plan
    pos, gam, sig0, sig, ref = sums
    live = int((gam != 0).any(1).sum())
    for tpl in (0, 1):
        for tr in (False, True):
            kw = dict(p=4, theta=1e-3, ncrit=ncrit, p2p_tpl=tpl, outputs=7 if tr else 3)
            if kind == "mixed":
                kw.update(sigma_rule=FMM_SIGMA_MIXED)
            plan = Plan(N, Params.default(**kw))
            sg = None if kind == "one" else to_dev(sig)
            u, s = plan.eval(to_dev(pos), to_dev(gam), sigma=sg, sigma_uniform=float(sig0))
            torch.cuda.synchronize()
            st = plan.stats()
            assert st.m2l_pairs == 0 and st.p2p_pairs == N * N
            assert st.p2p_pairs_near + st.p2p_pairs_mid + st.p2p_pairs_far == N * live
            ud, sd = ref[kind, tr]
            assert rel_l2(u.cpu().numpy(), ud) < 2e-5, (tpl, tr)
            assert rel_l2(s.cpu().numpy(), sd) < 5e-5, (tpl, tr)
            plan.close()


@pytest.mark.parametrize("kind", ["one", "each"])
@pytest.mark.parametrize("n", [1, 2, 31, 33, 63, 64, 65, 1023, 1025, 2049])
def test_direct_sum_at_tile_and_share_edges(n, kind):
    """The all-pairs kernel where a 64-target tile or a warp's 32nd of the
    sources is empty, partly filled or one past full, against the FP64 pair
    sum; rel-L2 2e-6 (u) and 5e-6 (s), the tolerances of the all-pairs parity
    test (FP32 unit roundoff times the growth of sums of a few thousand terms
    of exact differences)."""
    import torch
    from oracle import pairs
    from paper_1106_5273_gb300 import direct
    w = workloads.uniform_ball(n)
    sig = (w["sigma"] * np.linspace(0.7, 1.3, n)).astype(np.float32) if kind == "each" else None
    u, s = direct(to_dev(w["pos"]), to_dev(w["gamma"]), sigma=None if sig is None else to_dev(sig),
                  sigma_uniform=float(w["sigma"]))
    torch.cuda.synchronize()
    x, g = w["pos"].astype(np.float64), w["gamma"].astype(np.float64)
    sg = np.full(n, float(w["sigma"])) if sig is None else sig.astype(np.float64)
    ud, sd = pairs.pair_sum(x, g, x, g, sg, None, np.eye(n, dtype=bool))
    if n == 1:
        assert not u.cpu().numpy().any() and not s.cpu().numpy().any()
    else:
        assert rel_l2(u.cpu().numpy(), ud) < 2e-6
        assert rel_l2(s.cpu().numpy(), sd) < 5e-6
