"""lbm_autotune compares complete steps: every candidate runs with the ghost launch that its steps need.

The launches are counted with the profiler of torch.  On a grid with walls every kernel but the
double-float ones (which form the walls in their tiles) has one ghost launch a step.
"""
import numpy as np
import pytest

from paper_1305_4736_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

WALL, PER = (wl.BC_NEQ_WALL, 1.0, 0.02, 0.0, 1.01), (wl.BC_PERIODIC, 0, 0, 0, 0)


@pytest.fixture(scope="module")
def lbm():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_1305_4736_gb300 import build, lbm as L
    build.build()
    L.load()
    from torch.profiler import ProfilerActivity, profile
    with profile(activities=[ProfilerActivity.CUDA]):        # the first session sets the profiler up
        torch.ones(1, device="cuda").add_(1)
        torch.cuda.synchronize()
    return L


def _counts(f):
    import torch
    from torch.profiler import ProfilerActivity, profile
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        f()
        torch.cuda.synchronize()
    names = [e.name for e in prof.events() if "lbm::k_" in e.name]
    if not names:
        pytest.skip("the profiler records no launches here")
    return {k: sum(n.split("<")[0].endswith(k) for n in names)
            for k in ("k_ghost", "k_step", "k_step_tma", "k_step_tma_pipe", "k_step_stream", "k_step_dd")}


@pytest.mark.parametrize("edges,ghosts", [([PER, PER, WALL, WALL], "walls"), ([PER] * 4, "periodic")])
@pytest.mark.parametrize("precision", [0, 1])
def test_candidates_are_timed_with_their_ghost_launches(lbm, precision, edges, ghosts):
    p = wl.shear_layer(160, ny=64)
    p.bc = edges
    s = lbm.Solver.from_problem(p, precision=precision)
    s.init(*p.fields())
    s.step(2)
    state = s.get_state()
    reps = 3
    n = _counts(lambda: s.autotune(reps))
    assert n["k_step"] == 4 * (reps + 1) and n["k_step_tma"] == reps + 1 and n["k_step_stream"] == reps + 1
    if ghosts == "walls":
        assert n["k_ghost"] == n["k_step"] + n["k_step_tma"] + n["k_step_tma_pipe"] + n["k_step_stream"]
    else:                                   # only these two read filled ghost cells
        assert n["k_ghost"] == n["k_step_tma_pipe"] + n["k_step_stream"]
    assert np.array_equal(s.get_state(), state)
    s.close()
