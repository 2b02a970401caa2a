"""M2L steps of trees so deep that (tile, translation) does not fit a word with
42-cell tiles or a batch's key buckets (marked gpu), but does with tiles of 64
cells.  Two blobs that share a cell of level 15 are seen across the domain by
one blob alone in a cell of level 1, from a distance that only small cells
pass (5 sigma): 56 bits of translation.  With the few tiles of four blobs the
plain evaluation sorts whole words and the batch one part after the other; the
4100 cells of the lattice take 7 bits of 64-cell tiles and 8 of 42."""
import numpy as np
import pytest

from gpu_common import rel_l2, to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _cloud(m=0, level=16):
    side = 1.0 + 2.0 ** -10  # the free-space cube of the unit box
    lo, a = 0.5 - 0.5 * side, side * 2.0 ** (1 - level)
    k = np.floor(np.array([5.0 / 6.0, 11.0 / 12.0, 11.0 / 12.0]) * 2.0 ** (level - 1))
    near, far = lo + (k + 0.25) * a, lo + (k + 0.75) * a  # the two halves of a cell of level 15
    pts = [np.zeros((1, 3)), np.ones((1, 3)), near[None], far[None]]
    if m:  # an m^3 lattice outside the first octant
        i = (np.arange(m) + 0.3) / m
        x = np.stack(np.meshgrid(i, i, i, indexing="ij"), -1).reshape(-1, 3)
        pts.append(x[(x > 0.5).any(1)])
    pos = np.concatenate(pts).astype(np.float32)
    ca = lo + 0.25 * side
    d = np.linalg.norm(near - ca) - np.sqrt(3.0) * abs(ca)
    gam = np.random.default_rng(3).standard_normal(pos.shape).astype(np.float32)
    return pos, gam, float(np.float32((d - 2.0 ** (-level - 3)) / 5.0))


@pytest.mark.parametrize("mode", [1, 2])
def test_batch_matches_the_plain_evaluation(mode):
    import torch
    from paper_1106_5273_gb300 import Params, Plan
    pos, gam, sig = _cloud()
    n = len(pos)
    prm = Params.default(p=8, theta=0.5, ncrit=1, m2l_mode=mode)
    plain, batch = Plan(n, prm), Plan(3 * n, prm)
    u, s = plain.eval(to_dev(pos), to_dev(gam), sigma_uniform=sig)
    ub, sb = batch.eval_batch(np.arange(4) * n, to_dev(np.tile(pos, (3, 1))), to_dev(np.tile(gam, (3, 1))),
                              sigma_prob=np.full(3, sig, np.float32))
    torch.cuda.synchronize()
    a, b = plain.stats(), batch.stats()
    assert a.m2l_pairs > 0 and b.m2l_pairs == 3 * a.m2l_pairs and b.m2l_keys == a.m2l_keys
    for k in range(3):  # a few M2L terms per sum, each summed alone: FP32 rounding of the order
        assert rel_l2(ub[n * k:n * k + n].cpu(), u.cpu()) < 1e-6
        assert rel_l2(sb[n * k:n * k + n].cpu(), s.cpu()) < 1e-6


def test_lattice_with_42_cell_tiles():
    """Tensor-core against SIMT M2L: the tolerances of the parity tests."""
    import torch
    from paper_1106_5273_gb300 import Params, Plan
    pos, gam, sig = _cloud(16)
    out = []
    for mode in (1, 2):
        plan = Plan(len(pos), Params.default(p=8, theta=0.5, ncrit=1, m2l_mode=mode))
        u, s = plan.eval(to_dev(pos), to_dev(gam), sigma_uniform=sig)
        torch.cuda.synchronize()
        assert plan.stats().m2l_pairs > 1000
        out.append((u.cpu().numpy(), s.cpu().numpy()))
        plan.close()
    assert rel_l2(out[1][0], out[0][0]) < 1e-5 and rel_l2(out[1][1], out[0][1]) < 3e-5
