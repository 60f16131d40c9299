"""Half-stencil steps that exchange the position and velocity arrays (sets of
more than 65,536 slots, pairs of steps), in each way they are run: direct
launches (a length's first call), graphs (when it comes again), the timed steps
of profile(), and between the samples of a served set.  Against calls of one
step each, which take the plain step's kernels.

The half stencil's sums have no fixed order: forces differ by up to 1e-5 of
their RMS (about 100), which moves a velocity by 5e-6 and a position by less
than an ulp of the edge a step; five steps and the rounding of positions up to
41 (4e-6) stay within 2e-5 (positions) and 1e-4 (velocities)."""

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


def _one_by_one(box, nsteps):
    for _ in range(nsteps):
        box.step(1)


@pytest.mark.parametrize("nsteps", [2, 3, 5])
@pytest.mark.parametrize("L,n,force", [((26.0, 29.0, 31.0), 65537, {}),
                                       ((40.0, 36.3, 32.9), 140001, {"poiseuille_f": 0.1})])
def test_single_box(mods, L, n, force, nsteps):
    D, _ = mods
    x, v = uniform_box_state(L, n=n, seed=n)
    box, ref = (D.Box(L, seed=5, stencil=1, **force) for _ in range(2))
    ref.set_state(x, v)
    _one_by_one(ref, nsteps)
    want, stats = ref.get_state(), ref.stats()
    for advance in (box.step, box.step, box.profile):  # direct, graphs, timed
        box.set_state(x, v)
        advance(nsteps)
        _close(box.get_state(), want, L)
        st = box.stats()
        assert st["step"] == stats["step"] == nsteps and st["n"] == n
        assert st["virial"] == pytest.approx(stats["virial"], rel=1e-4)
    box.close()
    ref.close()


@pytest.mark.parametrize("nsteps", [2, 5])
def test_packed_boxes_some_stopped(mods, nsteps):
    _, B = mods
    rng = np.random.default_rng(3)
    Ls = [tuple(rng.uniform(6.0, 12.0, 3).round(1)) for _ in range(52)]
    n = [0 if k in (0, 17) else int(4 * np.prod(L)) + k for k, L in enumerate(Ls)]
    assert sum(n) > 131072
    empty = (np.zeros((0, 3), np.float32),) * 2
    states = [uniform_box_state(L, n=m, seed=m) if m else empty for L, m in zip(Ls, n)]
    descs = [B.make_desc(L, m, seed=k, steps=(0, 1, 4)[k % 3]) for k, (L, m) in
             enumerate(zip(Ls, n))]
    bt, ref = (B.Batch(descs, stencil=1) for _ in range(2))

    def load(b):
        for k, s in enumerate(states):
            b.set_state(k, *s)

    load(ref)
    _one_by_one(ref, nsteps)
    want = [ref.get_state(k) for k in range(len(Ls))]
    steps = [s["step"] for s in ref.stats()]
    assert steps[1:4] == [1, min(4, nsteps), nsteps]
    for advance in (bt.step, bt.step, bt.profile):  # direct, graphs, timed
        load(bt)
        advance(nsteps)
        assert [s["step"] for s in bt.stats()] == steps
        for k, L in enumerate(Ls):
            _close(bt.get_state(k), want[k], L)
    bt.close()
    ref.close()


@pytest.mark.parametrize("steps,every,chunk,samples", [
    (40, 5, 33, 4),    # a graph of 32 steps: samples behind either step of a pair
    (20, 11, 20, 1)])  # direct launches: behind step 11, the first of its pair
def test_sampled_half_stencil_set(mods, steps, every, chunk, samples):
    """A served set above 65,536 slots, sampled between its exchanging steps."""
    import paper_1911_04712_gb300.serve as S
    D, _ = mods
    sizes = [(28.2, 66000), (11.0, 4097)]
    states = [uniform_box_state(L, n=n, seed=n) for L, n in sizes]
    q = S.Queue(1 << 30, chunk_steps=chunk, sample_every=every, nbins=4, stencil=1)
    tk = [q.submit_state(S.make_request(L, n=n, seed=n, steps=steps), x, v)
          for (L, n), (x, v) in zip(sizes, states)]
    q.wait_all(300)
    got = [q.result(t) for t in tk]
    q.close()
    for (L, n), (x, v), g in zip(sizes, states, got):
        box = D.Box(L, seed=n, stencil=1)
        box.set_state(x, v)
        kT, pr = [], []
        for s in range(1, steps + 1):
            box.step(1)
            if s > steps // 2 and s % every == 0:
                st = box.stats()
                kT.append(st["kT"])
                pr.append(st["pressure"])
        box.close()
        assert g["samples"] == len(kT) == samples
        # 40 steps of sums in another order: velocities 1e-4 apart at random, which a
        # mean over 4,000 particles takes to 3e-6
        assert g["kT_mean"] == pytest.approx(np.mean(kT), rel=3e-5)
        assert g["pressure_mean"] == pytest.approx(np.mean(pr), rel=3e-5)
