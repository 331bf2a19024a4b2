"""Walls of the double-float float64 kernels are formed in float64.

With every rate 0, the upwind limiter and Courant number 1 for the fastest axis shell, a step takes the
value next to a wall to f0 - c (f0 - fg), c <= 1: that shell's populations become the ghost cell's value
fg.  Against the plain float64 kernel (step_kernel 1), whose walls a launch forms in float64: the split
rounds f0 and fg to 48 bits (2^-49), the difference, the product and the last difference round a low part
each (2^-49 of a value of at most twice the largest population or result): 2^-49 (2 + 3 * 2) = 2 * 2^-47 of
it.  Walls formed in double-float, some thirty operations on moments, are up to 4.5 * 2^-47 off.
"""
import numpy as np
import pytest

from paper_1305_4736_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

W1, W2 = (wl.BC_NEQ_WALL, 1.0, 0.02, 0.0, 1.01), (wl.BC_NEQ_WALL, 1.0, -0.03, 0.01, 0.99)


@pytest.fixture(scope="module")
def lbm():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_1305_4736_gb300 import build, lbm as L
    build.build()
    L.load()
    return L


def _solver(lbm, p, kernel, f):
    s = lbm.Solver.from_problem(p, step_kernel=kernel)
    s.set_state(f)
    return s


@pytest.mark.parametrize("seed", range(3))
@pytest.mark.parametrize("kernel,nx,ny", [(9, 64, 12), (9, 65, 5), (8, 64, 48), (8, 641, 515)])
def test_wall_ghosts_have_float64_accuracy_alone_and_batched(lbm, kernel, nx, ny, seed):
    p = wl.shear_layer(nx, ny=ny)
    p.bc = [W1, W2, W2, W1]
    p.s, p.Pr, p.limiter, p.dt = np.zeros(16), 1.0, 2, p.dx / 6.0
    f = np.random.default_rng(seed).uniform(0.5, 1.5, (16, ny, nx))
    plain, alone, member = (_solver(lbm, p, k, f) for k in (1, kernel, kernel))
    b = lbm.Batch([member])
    for s in (plain, alone, b):
        s.step(1)
    want, got, batched = plain.get_state(), alone.get_state(), member.get_state()
    b.close()
    assert np.array_equal(got, batched)
    assert np.abs(got - want).max() <= 2 * 2.0 ** -47 * max(np.abs(want).max(), np.abs(f).max())
    for s in (plain, alone, member):
        s.close()
