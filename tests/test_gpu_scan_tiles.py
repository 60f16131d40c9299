"""The cell scan at the edges of its tiles of 4096 entries (cells + 1): one
tile, a tile filled but for one entry, one entry in the next, several tiles;
empty boxes' worth of cells and crowded ones.  Forces through the scan
against those of the allocation-free call, which builds its cell list by a
scan of its own, within the contract's 1e-5 of their RMS."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("stencil", [0, 1])
@pytest.mark.parametrize("grid,n", [((3, 3, 3), 300), ((23, 11, 8), 9000), ((8, 16, 16), 2),
                                    ((8, 16, 16), 6000), ((7, 17, 17), 6000),
                                    ((16, 16, 16), 12000), ((12, 25, 27), 30000),
                                    ((3, 3, 900), 30000)])
def test_cell_starts_across_tiles(grid, n, stencil):
    torch = pytest.importorskip("torch")
    from paper_1911_04712_gb300 import build
    build.build()
    import paper_1911_04712_gb300.dpd as D
    L = tuple(g + 0.25 for g in grid)
    g = torch.Generator(device="cuda").manual_seed(n)
    x = torch.rand((n, 3), generator=g, device="cuda") * torch.tensor(L, device="cuda")
    x = torch.where(x >= torch.tensor(L, device="cuda"), torch.zeros_like(x), x)
    v = torch.randn((n, 3), generator=g, device="cuda")
    ref = D.forces_noalloc(x, v, L, seed=3).cpu().numpy()
    box = D.Box(L, seed=3, stencil=stencil)
    box.set_state(x, v)
    f = box.get_forces()
    f = f.cpu().numpy() if hasattr(f, "cpu") else f
    box.close()
    rms = max(float(np.sqrt((ref.astype(np.float64) ** 2).mean())), 1e-6)
    assert np.abs(f - ref).max() <= 1e-5 * rms
