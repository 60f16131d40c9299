"""Box.profile times the kernels that Box.step runs: kernel names of the L = 44
box's half-stencil steps, which exchange their arrays, by the profiler."""

import pytest

from paper_1911_04712_gb300.workloads import uniform_box_state

pytestmark = pytest.mark.gpu


def test_profile_times_the_kernels_that_steps_run():
    torch = pytest.importorskip("torch")
    from torch.profiler import ProfilerActivity, profile
    from paper_1911_04712_gb300 import build
    build.build()
    import paper_1911_04712_gb300.dpd as D
    box = D.Box(44.0, seed=1, stencil=1)
    box.set_state(*uniform_box_state(44.0, rho=3.0, seed=1))

    def kernels(advance):
        with profile(activities=[ProfilerActivity.CPU, ProfilerActivity.CUDA]) as p:
            advance(2)
            torch.cuda.synchronize()
        return sorted(e.key.split("(")[0] for e in p.key_averages() if "dpd::k_" in e.key)

    names = [kernels(f) for f in (box.step, box.profile, box.step, box.profile)][2:]
    box.close()
    if not names[0]:
        pytest.skip("no kernel names from the profiler here")
    assert names[0] == names[1] and any("k_kick_bin" in k for k in names[1])
