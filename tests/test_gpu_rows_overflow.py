"""Dense places in the row-parallel force kernels: targets whose neighbours
overflow a list or the queue are evaluated in rounds, row after row, each
round a share of every target's candidates.  Against the direct routine
(force variant 0): bit for bit with the full stencil, within the contract's
1e-5 of the force RMS with the half stencil, whose sums have no fixed order.

The drops: every candidate a neighbour (a round's queue filled to its last
place), many rounds a row, across faces and corners (a share that spans both
parts of a row), in boxes of either list length, whole blocks and a last one.
The time step is 1e-6 (and the noise small), so that the half stencil's states
stay comparable over the steps."""

import time

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


def _drop(L, n, m, size, centre, seed):
    """n particles, the first m of them in a cube of edge `size` about `centre`."""
    x, v = uniform_box_state(L, n=n, seed=seed)
    L = np.asarray(L, dtype=np.float64)
    d = (x[:m].astype(np.float64) / L - 0.5) * size + np.asarray(centre)
    x[:m] = (d - np.floor(d / L) * L).astype(np.float32)
    x[x >= L.astype(np.float32)] = 0.0
    return x, v


def _box(dpd, L, x, v, stencil, kind, variant):
    box = dpd.Box(L, kT=1e-4, dt=1e-6, seed=5, stencil=stencil, poiseuille_f=0.1, variant=variant,
                  noise=1 if kind == "gaussian" else None)
    if kind == "species":
        box.set_species(np.array([[25.0, 40.0], [40.0, 25.0]]), np.full((2, 2), 4.5),
                        np.array([[1.0, 0.8], [0.8, 0.9]]))
        box.set_state(x, v, species=(np.arange(len(x)) % 2).astype(np.int32))
    else:
        box.set_state(x, v)
    return box


CASES = [  # L, n, m, size, centre
    ((6.0, 5.0, 7.0), 400, 400, 0.4, (3.2, 2.2, 3.3)),   # all of them neighbours, short lists
    ((4.0, 4.2, 4.4), 700, 700, 0.5, (0.0, 0.0, 0.0)),   # at the corner; long lists
    ((9.0, 8.0, 10.0), 2500, 1500, 3.0, (0.1, 4.0, 9.8)),  # 55 a cell, across faces
    ((12.0, 3.5, 3.2), 1801, 900, 2.5, (11.9, 1.0, 0.2)),
    ((7.0, 7.0, 7.0), 33, 33, 0.2, (3.5, 0.0, 3.5)),
    ((12.0, 12.0, 12.0), 13001, 9000, 5.0, (6.0, 6.0, 0.0)),  # 72 a cell, long lists
]


@pytest.mark.parametrize("stencil", [0, 1])
@pytest.mark.parametrize("kind", ["plain", "gaussian", "species"])
@pytest.mark.parametrize("L,n,m,size,centre", CASES)
def test_dense_places_equal_the_direct_routine(dpd, L, n, m, size, centre, kind, stencil):
    x, v = _drop(L, n, m, size, centre, n)
    out = []
    for variant in (None, 0):
        box = _box(dpd, L, x, v, stencil, kind, variant)
        out.append([box.get_forces()])
        box.step(3)
        out[-1] += [box.get_forces(), box.get_state()[1]]
        box.close()
    got, ref = out
    rms = max(float(np.sqrt((ref[0].astype(np.float64) ** 2).sum(1).mean())), 1e-3)
    for g, r, tol in zip(got, ref, (FORCE_TOL * rms, 10 * FORCE_TOL * rms, FORCE_TOL)):
        if stencil == 0:
            assert np.array_equal(g, r)
        else:
            assert np.abs(g.astype(np.float64) - r).max() <= tol


def test_allocation_free_forces_at_dense_places(dpd):
    torch = pytest.importorskip("torch")
    for L, n, m, size, centre in CASES:
        x, v = _drop(L, n, m, size, centre, n)
        box = dpd.Box(L, seed=5, variant=0)
        box.set_state(x, v)
        ref = box.get_forces()
        box.close()
        f = dpd.forces_noalloc(torch.from_numpy(x).cuda(), torch.from_numpy(v).cuda(), L, seed=5)
        assert np.array_equal(f.cpu().numpy(), ref)


@pytest.mark.parametrize("stencil,n", [(0, 40000), (0, 65000), (1, 65000), (1, 260000)])
def test_a_drop_is_not_slower_than_on_the_direct_routine(dpd, stencil, n):
    """All particles in a drop of 15 a cell: the kernels that such a box runs
    against the tuned direct kernel."""
    torch = pytest.importorskip("torch")
    L = (n / 3.0) ** (1 / 3)
    x, v = _drop((L,) * 3, n, n, (n / 15.0) ** (1 / 3), (L / 2,) * 3, 7)
    took = {}
    for variant in (None, "direct"):
        if variant:
            variant = int(box.get_param(dpd.PARAM_FORCE_VARIANT))  # noqa: F821
            box.close()  # noqa: F821
        box = _box(dpd, (L,) * 3, x, 0 * v, stencil, "plain", variant)
        box.step(32)
        torch.cuda.synchronize()
        took[variant] = min(_time(torch, box) for _ in range(5))
    box.close()
    rows, direct = took.values()
    assert rows < 1.2 * direct, (rows, direct)


def _time(torch, box):
    t = time.perf_counter()
    box.step(32)
    torch.cuda.synchronize()
    return time.perf_counter() - t
