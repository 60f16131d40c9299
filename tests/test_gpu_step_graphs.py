"""A call of n steps replays graphs of 32 and of 2^k steps (small sets); any
split of the same steps into calls gives the same bits (full stencil)."""

import numpy as np
import pytest

from paper_1911_04712_gb300.workloads import uniform_box_state

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dpd():
    from paper_1911_04712_gb300 import build
    build.build()
    import paper_1911_04712_gb300.dpd as d
    return d


@pytest.mark.parametrize("n", [135, 131072, 131073])
def test_calls_of_any_length_give_the_same_bits(dpd, n):
    L = 3.0 if n < 1000 else 36.0
    x, v = uniform_box_state(L, n=n, seed=9)
    splits = [[2, 3, 15, 31], [51], [33, 18], [16, 8, 4, 2, 1, 20], [1] * 3 + [48]]
    outs = []
    for calls in splits:
        box = dpd.Box(L, seed=4)
        box.set_state(x, v)
        for k in calls:
            box.step(k)
        outs.append((*box.get_state(), box.get_forces(), np.array([box.stats()["step"]])))
        box.close()
    for out in outs[1:]:
        for a, b in zip(out, outs[0]):
            assert np.array_equal(a, b)
