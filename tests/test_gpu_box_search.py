"""The warp-wide search for a packed set's box of a slot, on sets whose box
count lies on both sides of a round of 32 probes (one round up to 32 boxes,
two up to 1024, three above), with empty boxes and boxes of fewer slots than
a warp: every box against the same box in a set of its own.  The full
stencil's sums have a fixed order, so the results are the same bits."""

import numpy as np
import pytest

from paper_1911_04712_gb300.workloads import uniform_box_state

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def batch():
    from paper_1911_04712_gb300 import build
    build.build()
    import paper_1911_04712_gb300.batch as B
    return B


def _run(B, picks, states, nst):
    bt = B.Batch([B.make_desc(3.0, len(states[k][0]), seed=k) for k in picks], stencil=0)
    for j, k in enumerate(picks):
        bt.set_state(j, *states[k])
    bt.step(nst)
    out = [(bt.get_state(j), bt.get_forces(j)) for j in range(len(picks))]
    st = [(s["n"], s["step"]) for s in bt.stats()]
    bt.close()
    return out, st


@pytest.mark.parametrize("nbox", [2, 31, 32, 33, 1023, 1024, 1025, 2100])
def test_every_box_of_a_set_is_found(batch, nbox):
    sizes = np.random.default_rng(nbox).choice([0, 1, 5, 31, 32, 33, 64, 81], nbox)
    sizes[-1] = 5
    empty = (np.zeros((0, 3), np.float32),) * 2
    states = [uniform_box_state(3.0, n=int(n), seed=k) if n else empty
              for k, n in enumerate(sizes)]
    nst = 3
    got, st = _run(batch, range(nbox), states, nst)
    assert [s[0] for s in st] == list(sizes)
    rng = np.random.default_rng(1)
    for k in sorted({0, nbox - 1, *rng.integers(0, nbox, 40)}):
        if sizes[k] == 0:
            continue
        (ref,), _ = _run(batch, [k], states, nst)
        for a, b in zip((*got[k][0], got[k][1]), (*ref[0], ref[1])):
            np.testing.assert_array_equal(a, b, err_msg=f"box {k} of {nbox}")
