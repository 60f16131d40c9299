"""The row-parallel force kernels that small single boxes run by default,
against the direct routine (force variant 0, which the parity tests hold
against the FP64 oracle): bit for bit with the full stencil, within the
contract's 1e-5 of the force RMS with the half stencil, whose sums have no
fixed order.  Sizes at the edges of a block of 32 targets, boxes whose rows
wrap, the largest boxes of the rule and one past it, and a dense place that
overflows a row's list."""

import numpy as np
import pytest

from paper_1911_04712_gb300.workloads import uniform_box_state

pytestmark = pytest.mark.gpu

FORCE_TOL = 1e-5


@pytest.fixture(scope="module")
def dpd():
    from paper_1911_04712_gb300 import build
    build.build()
    import paper_1911_04712_gb300.dpd as d
    return d


def _run(dpd, L, x, v, stencil, kind, variant):
    box = dpd.Box(L, seed=5, stencil=stencil, poiseuille_f=0.1, variant=variant,
                  noise=1 if kind == "gaussian" else None)
    if kind == "species":
        a = np.array([[25.0, 40.0], [40.0, 25.0]])
        g = np.full((2, 2), 4.5)
        rc = np.array([[1.0, 0.8], [0.8, 0.9]])
        box.set_species(a, g, rc)
        box.set_state(x, v, species=(np.arange(len(x)) % 2).astype(np.int32))
    else:
        box.set_state(x, v)
    first = box.get_forces()
    box.step(3)
    out = first, box.get_forces(), box.get_state()[1], box.stats()["virial"]
    box.close()
    return out


CASES = [((3.0, 3.0, 3.0), 1), ((3.0, 3.0, 3.0), 31), ((3.0, 3.4, 3.9), 33),
         ((5.0, 6.5, 7.25), 707), ((40.0, 3.0, 3.5), 97), ((8.0, 8.0, 8.0), 6144),
         ((26.0, 26.0, 26.0), 65536), ((26.0, 26.0, 26.0), 65537),
         ((8.0, 9.0, 10.0), 5041), ((8.0, 9.0, 10.0), 8640)]  # long lists; 12 per cell


@pytest.mark.parametrize("stencil", [0, 1])
@pytest.mark.parametrize("kind", ["plain", "gaussian", "species"])
@pytest.mark.parametrize("L,n", CASES)
def test_rows_equal_the_direct_routine(dpd, L, n, kind, stencil):
    x, v = uniform_box_state(L, n=n, seed=n)
    _compare(dpd, L, x, v, stencil, kind)


@pytest.mark.parametrize("stencil", [0, 1])
def test_rows_fall_back_where_a_list_overflows(dpd, stencil):
    L = (12.0, 11.0, 10.0)
    x, v = uniform_box_state(L, n=4000, seed=3)
    x[:400] = 5.5 + (x[:400] / np.float32(12.0) - np.float32(0.5))  # 400 particles in one cell's size
    _compare(dpd, L, x, v, stencil, "plain")


@pytest.mark.parametrize("L,n", [((3.0, 3.0, 3.0), 1), ((3.0, 4.5, 3.2), 31), ((6.0, 6.5, 7.0), 819),
                                 ((31.0, 31.0, 34.0), 32768), ((8.0, 8.0, 8.0), 32768)])
def test_allocation_free_forces_equal_the_direct_routine(dpd, L, n):
    import torch
    x, v = uniform_box_state(L, n=n, seed=n + 1)
    box = dpd.Box(L, seed=5, variant=0)
    box.set_state(x, v)
    ref = box.get_forces()
    box.close()
    for _ in range(2):  # the second call finds the scratch as the first left it
        f = dpd.forces_noalloc(torch.from_numpy(x).cuda(), torch.from_numpy(v).cuda(), L, seed=5)
        assert np.array_equal(f.cpu().numpy(), ref)


def _compare(dpd, L, x, v, stencil, kind):
    got = _run(dpd, L, x, v, stencil, kind, None)
    ref = _run(dpd, L, x, v, stencil, kind, 0)
    rms = max(float(np.sqrt((ref[0].astype(np.float64) ** 2).sum(1).mean())), 1e-3)
    if stencil == 0:
        for g, r in zip(got, ref):
            assert np.array_equal(g, r)
    else:
        assert np.abs(got[0].astype(np.float64) - ref[0]).max() <= FORCE_TOL * rms
        # three steps later the states differ by the rounding of the sums
        assert np.abs(got[1].astype(np.float64) - ref[1]).max() <= 10 * FORCE_TOL * rms
        assert np.abs(got[2].astype(np.float64) - ref[2]).max() <= 3 * 0.005 * FORCE_TOL * rms


@pytest.mark.parametrize("n", [700, 131000])
@pytest.mark.parametrize("stencil", [0, 1])
def test_noise_changed_on_a_loaded_box(dpd, n, stencil):
    """The force kernel follows the noise: a box whose noise is changed after
    loading steps as one that had it from the start."""
    L = 6.0 if n < 1000 else 36.0
    x, v = uniform_box_state(L, n=n, seed=2)
    for before, after in ((0, 1), (1, 0)):
        out = []
        for first in (before, after):
            box = dpd.Box(L, seed=8, stencil=stencil, noise=first)
            box.set_state(x, v)
            box.set_param(dpd.PARAM_NOISE, after)
            box.set_state(x, v)
            out.append(box.get_forces())
            box.close()
        rms = float(np.sqrt((out[1].astype(np.float64) ** 2).sum(1).mean()))
        err = np.abs(out[0].astype(np.float64) - out[1]).max()
        assert err <= (0.0 if stencil == 0 else FORCE_TOL * rms)
