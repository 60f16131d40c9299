"""Steps enqueued on a stream that the caller is capturing become nodes of the
caller's graph, whatever their number: calls of one step and of whole chunks of
32 too, which otherwise replay graphs of the engine's own.  Replaying the
captured graph gives the bits of the same steps outside a capture (full
stencil)."""

import numpy as np
import pytest

from paper_1911_04712_gb300.workloads import uniform_box_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("before", [0, 33])  # steps before the capture: engine graphs made, or not
@pytest.mark.parametrize("nsteps", [1, 5, 32, 40])
def test_steps_in_a_callers_capture(nsteps, before):
    torch = pytest.importorskip("torch")
    from paper_1911_04712_gb300 import build
    build.build()
    import paper_1911_04712_gb300.dpd as D
    L = (6.0, 5.0, 7.5)
    x, v = uniform_box_state(L, n=700, seed=3)
    out = []
    for captured in (True, False):
        box = D.Box(L, seed=4)
        stream = torch.cuda.Stream()
        box.set_stream(stream)
        box.set_state(x, v)
        box.step(before)
        if captured:
            stream.synchronize()
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=stream):
                box.step(nsteps)
            with torch.cuda.stream(stream):
                graph.replay()
        else:
            box.step(nsteps)
        out.append((*box.get_state(), box.get_forces()))
        box.step(2)  # the engine's own graphs still serve the box
        out[-1] += box.get_state()
        box.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b)
