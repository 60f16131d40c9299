"""Sampling behind fused steps: the accumulators of served runs, whose samples
fall inside chunks and at their ends, against the same runs in boxes of their
own with plain steps, read out at the sampled steps.  The full stencil's
trajectories are the same bits; the statistics sum v^2 in FP32 pairs there
and in FP64 here, which leaves a rounding of each particle's v^2 (6e-8, and
less in the mean): 1e-6 relative."""

import numpy as np
import pytest

from paper_1911_04712_gb300.workloads import uniform_box_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("chunk", [40, 33, 7])
def test_samples_equal_plain_runs_read_out(chunk):
    from paper_1911_04712_gb300 import build
    build.build()
    import paper_1911_04712_gb300.dpd as D
    import paper_1911_04712_gb300.serve as S
    steps, every = 40, 8
    # one work item, two (4097 particles), several; two particles
    sizes = [(4.0, 200), (11.0, 4097), (15.5, 11000), (3.0, 2)]
    states = [uniform_box_state(L, n=n, seed=n) for L, n in sizes]
    q = S.Queue(1 << 30, chunk_steps=chunk, sample_every=every, nbins=4)
    tk = [q.submit_state(S.make_request(L, n=n, seed=n, steps=steps), x, v, keep_final=True)
          for (L, n), (x, v) in zip(sizes, states)]
    q.wait_all(300)
    got = [q.result(t) for t in tk]
    fin = [q.final_state(t, n) for t, (_, n) in zip(tk, sizes)]
    q.close()
    for (L, n), (x, v), g, f in zip(sizes, states, got, fin):
        box = D.Box(L, seed=n)
        box.set_state(x, v)
        kT, pr = [], []
        for s in range(every, steps + 1, every):
            box.profile(every)  # plain steps
            if s > steps // 2:
                st = box.stats()
                kT.append(st["kT"])
                pr.append(st["pressure"])
        ref = box.get_state()
        box.close()
        assert g["samples"] == len(kT) == 3
        assert g["kT_mean"] == pytest.approx(np.mean(kT), rel=1e-6)
        assert g["pressure_mean"] == pytest.approx(np.mean(pr), rel=1e-6)
        for a, b in zip(f, ref):
            np.testing.assert_array_equal(a, b)
