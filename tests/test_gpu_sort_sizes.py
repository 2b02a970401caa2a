"""The Morton sort at the edges of its tiles (marked gpu): one tile, a tile
exactly full and one past it, the sizes where the keys per thread change,
keys that vary in few digits and in all; sorted keys and order are those of a
stable sort, bit for bit."""
import numpy as np
import pytest

from gpu_common import to_dev

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("kind", ["random", "few"])
@pytest.mark.parametrize("n", [1, 2, 33, 1023, 1024, 1025, 65535, 65536, 65537, (1 << 20), (1 << 20) + 1, 1500007])
def test_order_is_the_stable_order_of_the_keys(n, kind):
    import torch
    from oracle import tree as otree
    from paper_1106_5273_gb300 import Params, Plan
    g = np.random.default_rng(n)
    pos = g.random((n, 3))
    if kind == "few":  # 4 cells per axis of the unit cube: two key digits vary, most keys are equal
        pos = (np.floor(pos * 4) + 0.5) / 4
    pos = pos.astype(np.float32)
    keys = otree.interleave(otree.quantize(pos, np.zeros(3), 1.0))
    # one leaf per particle cluster is enough: large leaves keep the rest of the evaluation small
    plan = Plan(n, Params.default(p=1, theta=0.9, ncrit=4096, periodic=1, images=1, box_min=(0, 0, 0), box_len=1.0,
                                  m2l_mode=1))
    zero = torch.zeros((n, 3), device="cuda")
    for _ in range(2):
        plan.eval(to_dev(pos), zero, sigma_uniform=1e-4, stretching=False)
        torch.cuda.synchronize()
        order, skeys = plan.order()
        want = np.argsort(keys, kind="stable")
        assert np.array_equal(skeys, keys[want]) and np.array_equal(order.astype(np.int64), want)
    plan.close()
