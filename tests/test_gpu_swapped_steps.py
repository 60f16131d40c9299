"""Half-stencil steps that exchange the position and velocity arrays (sets of
more than 65,536 slots, pairs of steps) against the plain step, which the
timed steps of profile() take: even and odd numbers of steps, launched
directly (a length's first call) and replayed, sets at the rule's edge, a
constant and a periodic force, packed sets with stopped and empty boxes.

The half stencil's sums have no fixed order: forces differ by up to 1e-5 of
their RMS (about 100), which moves a velocity by 5e-6 and a position by less
than an ulp of the edge a step; five steps and the rounding of positions up
to 41 (4e-6) stay within 2e-5 (positions) and 1e-4 (velocities)."""

import numpy as np
import pytest

from paper_1911_04712_gb300.workloads import uniform_box_state

pytestmark = pytest.mark.gpu

X_TOL, V_TOL = 2e-5, 1e-4


@pytest.fixture(scope="module")
def mods():
    from paper_1911_04712_gb300 import build
    build.build()
    import paper_1911_04712_gb300.batch as B
    import paper_1911_04712_gb300.dpd as D
    return D, B


def _close(a, b, L):
    d = a[0].astype(np.float64) - b[0]
    d -= np.round(d / L) * np.asarray(L)
    assert np.abs(d).max(initial=0.0) < X_TOL
    assert np.abs(a[1] - b[1]).max(initial=0.0) < V_TOL


@pytest.mark.parametrize("nsteps", [1, 2, 3, 5])
@pytest.mark.parametrize("L,n,force", [((26.0, 29.0, 31.0), 65537, {}),
                                       ((26.0, 29.0, 31.0), 65536, {}),
                                       ((40.0, 26.3, 30.9), 100001, {"poiseuille_f": 0.1})])
def test_single_box(mods, L, n, force, nsteps):
    D, _ = mods
    x, v = uniform_box_state(L, n=n, seed=n)
    boxes = [D.Box(L, seed=5, stencil=1, **force) for _ in range(2)]
    for _ in range(2):  # a new state each: direct launches first, then graphs
        for b in boxes:
            b.set_state(x, v)
        boxes[0].step(nsteps)
        boxes[1].profile(nsteps)
        _close(boxes[0].get_state(), boxes[1].get_state(), L)
        st = [b.stats() for b in boxes]
        assert st[0]["step"] == st[1]["step"] and st[0]["n"] == n
        assert st[0]["virial"] == pytest.approx(st[1]["virial"], rel=1e-4)
    for b in boxes:
        b.close()


@pytest.mark.parametrize("nsteps", [2, 5])
def test_packed_boxes_some_stopped(mods, nsteps):
    _, B = mods
    rng = np.random.default_rng(3)
    Ls = [tuple(rng.uniform(6.0, 12.0, 3).round(1)) for _ in range(40)]
    n = [0 if k in (0, 17) else int(4 * np.prod(L)) + k for k, L in enumerate(Ls)]
    assert sum(n) > 65536
    empty = (np.zeros((0, 3), np.float32),) * 2
    states = [uniform_box_state(L, n=m, seed=m) if m else empty for L, m in zip(Ls, n)]
    descs = [B.make_desc(L, m, seed=k, steps=(0, 1, 4)[k % 3]) for k, (L, m) in
             enumerate(zip(Ls, n))]
    out = []
    for advance in ("step", "profile"):
        bt = B.Batch(descs, stencil=1)
        for k, s in enumerate(states):
            bt.set_state(k, *s)
        getattr(bt, advance)(nsteps)
        out.append([bt.get_state(k) for k in range(len(Ls))])
        steps = [s["step"] for s in bt.stats()]
        bt.close()
    assert steps[1:4] == [1, min(4, nsteps), nsteps]
    for k, L in enumerate(Ls):
        _close(out[0][k], out[1][k], L)
