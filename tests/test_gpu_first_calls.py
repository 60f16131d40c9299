"""Which calls of several steps make graphs of the engine's own.  Graphs cost
their capture, so a set launches directly until a number of steps comes again,
and starts anew when its graphs were dropped (a changed parameter, a new
layout).

To see it, the calls run while another stream of this thread is being captured:
CUDA refuses to instantiate a graph then, so that a call that wants a new one
fails and a call of direct launches does not."""

import pytest

from paper_1911_04712_gb300.workloads import uniform_box_state

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dpd():
    pytest.importorskip("torch")
    from paper_1911_04712_gb300 import build
    build.build()
    import paper_1911_04712_gb300.dpd as d
    return d


def _step_without_new_graphs(box, nsteps):
    import torch
    graph, other = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    buf = torch.zeros(8, device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.graph(graph, stream=other, capture_error_mode="thread_local"):
        buf.add_(1.0)
        box.step(nsteps)
    box.stats()


def _box(dpd, n, stencil):
    import torch
    L = (n / 3.0) ** (1 / 3)
    box = dpd.Box(L, seed=1, stencil=stencil)
    stream = torch.cuda.Stream()  # the legacy stream may not run beside a capture
    box.set_stream(stream)
    box.set_state(*uniform_box_state(L, n=n, seed=2))
    return box, L


@pytest.mark.parametrize("stencil", [0, 1])
@pytest.mark.parametrize("n", [131200, 700, 66000])
def test_sets_capture_when_a_length_comes_again(dpd, n, stencil):
    box, L = _box(dpd, n, stencil)
    _step_without_new_graphs(box, 5)
    for change in (lambda: box.set_param(dpd.PARAM_BODYFORCE, 0.1),
                   lambda: box.set_state(*uniform_box_state(L, n=n + 1, seed=2))):
        box.step(5)  # captures
        _step_without_new_graphs(box, 5)  # replays
        change()
        _step_without_new_graphs(box, 5)  # as a first call
    box.close()
