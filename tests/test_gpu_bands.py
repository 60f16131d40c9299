"""Force launches of a packed set whose boxes need different general kernels
(Gaussian noise, several species, both): neighbours share a launch whatever
their kinds, as they do when all are of one kind, and the results are those of
the boxes alone (full stencil: the same bits)."""

import ctypes

import numpy as np
import pytest

from paper_1911_04712_gb300.workloads import uniform_box_state

pytestmark = pytest.mark.gpu

TABLES = (np.array([[25.0, 40.0], [40.0, 25.0]]), np.full((2, 2), 4.5),
          np.array([[1.0, 0.8], [0.8, 0.9]]))


def _batch(B, kinds, stencil):
    """Boxes plain (p), Gaussian (g), of two species (s), or both (b)."""
    descs = [B.make_desc(4.0 + 0.1 * (i % 3), 190 + i, seed=i, noise=int(k in "gb"),
                         species=TABLES if k in "sb" else None) for i, k in enumerate(kinds)]
    bt = B.Batch(descs, stencil=stencil)
    for i, k in enumerate(kinds):
        x, v = uniform_box_state(descs[i].box[0], n=190 + i, seed=i)
        bt.set_state(i, x, v, species=(np.arange(190 + i) % 2).astype(np.int32)
                     if k in "sb" else None)
    return bt, descs


def _kernels_per_step(torch, bt):
    """Kernel nodes of one step captured from a stream."""
    from paper_1911_04712_gb300.dpd import _stream_ptr, check, lib
    with open("/proc/self/maps") as f:
        rt = ctypes.CDLL(next(q.split()[-1] for q in f if "libcudart" in q))
    stream = torch.cuda.Stream()
    check(lib().dpd_batch_set_stream(bt._b, _stream_ptr(stream)))
    bt.step(0)
    torch.cuda.synchronize()
    s, graph, n = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p(), ctypes.c_size_t()
    assert rt.cudaStreamBeginCapture(s, 1) == 0  # thread-local
    try:
        bt.step(1)
    finally:
        rt.cudaStreamEndCapture(s, ctypes.byref(graph))
    assert graph.value and rt.cudaGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    rt.cudaGraphDestroy(graph)
    return n.value


@pytest.mark.parametrize("stencil", [0, 1])
@pytest.mark.parametrize("kinds", ["gs" * 3, "gsb" * 4, "ppp" + "gs" * 2, "gggsss"])
def test_kinds_share_a_launch(kinds, stencil):
    torch = pytest.importorskip("torch")
    from paper_1911_04712_gb300 import build
    build.build()
    import paper_1911_04712_gb300.batch as B
    import paper_1911_04712_gb300.dpd as D
    launches = []
    for ks in (kinds, kinds.replace("s", "g").replace("b", "g")):
        bt, descs = _batch(B, ks, stencil)
        launches.append(_kernels_per_step(torch, bt))
        if ks == kinds:
            bt2, _ = _batch(B, ks, stencil)
            bt2.step(3)
            got = [bt2.get_forces(i) for i in range(len(kinds))]
            bt2.close()
        bt.close()
    assert launches[0] == launches[1]
    for i, k in enumerate(kinds):
        box = D.Box(descs[i].box[0], seed=i, stencil=stencil, noise=int(k in "gb"), variant=0)
        x, v = uniform_box_state(descs[i].box[0], n=190 + i, seed=i)
        if k in "sb":
            box.set_species(*TABLES)
            box.set_state(x, v, species=(np.arange(190 + i) % 2).astype(np.int32))
        else:
            box.set_state(x, v)
        box.step(3)
        ref = box.get_forces()
        box.close()
        rms = float(np.sqrt((ref.astype(np.float64) ** 2).sum(1).mean()))
        # half stencil: sums without a fixed order, three steps apart
        tol = 0.0 if stencil == 0 else 1e-4 * rms
        assert np.abs(got[i].astype(np.float64) - ref).max() <= tol
