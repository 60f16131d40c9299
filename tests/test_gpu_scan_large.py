"""The cell scan on both sides of 2048 tiles (8,388,608 entries), above which a
block of its own scans the tiles' sums: sparse boxes of 161 x 161 cells, with
particles anywhere, crowded at the corner that all faces share and in the last
cells.  Forces against the oracle within the contract's 1e-5 of their RMS."""

import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("stencil", [0, 1])
@pytest.mark.parametrize("Lz", [161.25, 161.9, 163.25])  # 2038, 2038 and 2064 tiles
def test_forces_beyond_2048_tiles(Lz, stencil):
    from paper_1911_04712_gb300 import build
    build.build()
    import paper_1911_04712_gb300.dpd as D
    L = np.array([161.25, 161.25, Lz])
    rng = np.random.default_rng(int(Lz * 100))
    last = L - 0.75  # the last cells
    x = np.concatenate([rng.uniform(0.0, 1.0, (2000, 3)) * L,
                        rng.uniform(-2.5, 2.5, (900, 3)),
                        last + rng.uniform(-0.5, 0.74, (300, 3)),
                        rng.uniform(-2.0, 2.0, (500, 3)) + np.array([80.0, 0.0, L[2] / 2])])
    x = (x - np.floor(x / L) * L).astype(np.float32)
    x[x >= L.astype(np.float32)] = 0.0
    v = rng.normal(size=x.shape).astype(np.float32)
    box = D.Box(tuple(L), seed=3, stencil=stencil)
    box.set_state(x, v)
    f = box.get_forces()
    box.step(2)  # rebuilt from the cleared counts
    assert box.stats()["n"] == len(x)
    box.set_state(x, v)
    again = box.get_forces()
    box.close()
    # the edges as the kernels hold them, in FP32: 161.9 is not representable, and
    # its rounding (8e-6) alone moves forces across a face by 9.6e-3
    edges = tuple(L.astype(np.float32).astype(np.float64))
    p = O.Params(L=edges, a=25.0, gamma=4.5, kT=1.0, rc=1.0, dt=0.005, seed=3)
    ref, _ = O.forces(p, x, v, 0)
    rms = float(np.sqrt((ref ** 2).sum(1).mean()))
    for g in (f, again):
        assert np.abs(g.astype(np.float64) - ref).max() <= 1e-5 * rms
