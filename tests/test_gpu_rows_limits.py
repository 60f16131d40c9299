"""Which single boxes the row-parallel force kernels serve.  At each line of the
rule, by slots per cell and kind, and one slot past it: forces against the
direct routine (force variant 0), bit for bit with the full stencil, within the
contract's 1e-5 of the force RMS with the half stencil.  And on neither side may
a box be slower than on the tuned direct kernel: sparse boxes of many particles
were, when the lines did not look at the density."""

import time

import numpy as np
import pytest

from paper_1911_04712_gb300.workloads import uniform_box_state

pytestmark = pytest.mark.gpu

FULL = {"plain": [(1.7, 57344), (3.0, 65536), (4.9, 65536), (6.0, 106496), (8.0, 90112),
                  (11.0, 106496)],
        "gaussian": [(1.7, 57344), (3.0, 90112), (4.9, 90112), (6.0, 139264), (11.0, 139264)],
        "species": [(1.7, 57344), (3.0, 73728), (4.9, 90112), (8.0, 139264)]}
HALF = [(1.7, 90112), (3.0, 262144), (11.0, 262144)]
LINES = ([(0, k, r, n) for k in FULL for r, n in FULL[k]]
         + [(1, k, r, n) for k in FULL for r, n in HALF])


@pytest.fixture(scope="module")
def dpd():
    from paper_1911_04712_gb300 import build
    build.build()
    import paper_1911_04712_gb300.dpd as d
    return d


def _box(dpd, L, x, v, stencil, kind, variant):
    box = dpd.Box(L, seed=5, stencil=stencil, variant=variant, noise=int(kind == "gaussian"))
    if kind == "species":
        box.set_species(np.array([[25.0, 40.0], [40.0, 25.0]]), np.full((2, 2), 4.5),
                        np.array([[1.0, 0.8], [0.8, 0.9]]))
        box.set_state(x, v, species=(np.arange(len(x)) % 2).astype(np.int32))
    else:
        box.set_state(x, v)
    return box


def _edges(per_cell, n):
    """A box of n particles at about per_cell slots per cell (and no more)."""
    nc = int((n / per_cell) ** (1 / 3))
    a, b = nc, nc
    return (float(int(-(-n // (per_cell * a * b)))), float(a), float(b))


@pytest.mark.parametrize("past", [0, 1])
@pytest.mark.parametrize("stencil,kind,per_cell,n", LINES)
def test_both_sides_of_a_line(dpd, stencil, kind, per_cell, n, past):
    L = _edges(per_cell, n + past)
    x, v = uniform_box_state(L, n=n + past, seed=7)
    out = []
    for variant in (None, 0):
        box = _box(dpd, L, x, v, stencil, kind, variant)
        out.append(box.get_forces())
        box.close()
    got, ref = out
    if stencil == 0:
        assert np.array_equal(got, ref)
    else:
        rms = float(np.sqrt((ref.astype(np.float64) ** 2).sum(1).mean()))
        assert np.abs(got.astype(np.float64) - ref).max() <= 1e-5 * rms


@pytest.mark.parametrize("stencil,kind,per_cell,n", [
    (0, "plain", 1.0, 65000), (0, "gaussian", 1.0, 88000), (0, "species", 1.0, 88000),
    (0, "species", 2.0, 86000), (1, "plain", 1.0, 240000), (1, "species", 1.0, 240000)])
def test_sparse_boxes_are_not_slower_than_on_the_direct_kernel(dpd, stencil, kind, per_cell, n):
    torch = pytest.importorskip("torch")
    L = _edges(per_cell, n)
    x, v = uniform_box_state(L, n=n, seed=7)
    boxes = [_box(dpd, L, x, v, stencil, kind, None)]
    tuned = int(boxes[0].get_param(dpd.PARAM_FORCE_VARIANT))
    boxes.append(_box(dpd, L, x, v, stencil, kind, tuned))
    best = [1e9, 1e9]
    for _ in range(8):
        for k, box in enumerate(boxes):
            torch.cuda.synchronize()
            t = time.perf_counter()
            box.step(64)
            torch.cuda.synchronize()
            best[k] = min(best[k], time.perf_counter() - t)
    for box in boxes:
        box.close()
    assert best[0] < 1.05 * best[1], best
