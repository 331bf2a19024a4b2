"""The limited slope of the double-float float64 kernels where neighbouring differences nearly cancel.

At an extremum that is symmetric to some eight digits, the differences a and b of a cell to its
neighbours have opposite signs and a + b is of the size of their low float32 parts: the MC slope there
is zero, not a + b.  Every rate is zero, so a step is the convection alone: f less c_x and c_y (both
below 1) times flux differences whose terms are the differences and h/2 <= 1/4 times slopes.  Against the
float64 tile kernel (step_kernel 2): the split keeps 48 bits (2^-49 of a population), the result's
operations, fewer than 16 on terms of at most the largest population, round at 2^-47 each.  A slope that
is off by a + b would show as some 1e-9 of it.
"""
import numpy as np
import pytest

from paper_1305_4736_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lbm():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_1305_4736_gb300 import build, lbm as L
    build.build()
    L.load()
    return L


def _step(lbm, p, kernel, f):
    s = lbm.Solver.from_problem(p, step_kernel=kernel)
    s.set_state(f)
    s.step(1)
    out = s.get_state()
    s.close()
    return out


@pytest.mark.parametrize("eps", [1e-6, 1e-8, 1e-10, 1e-13])
@pytest.mark.parametrize("kernel,nx,ny", [(8, 64, 48), (8, 640, 512), (9, 64, 12)])
def test_slope_is_zero_where_differences_cancel(lbm, kernel, nx, ny, eps):
    p = wl.shear_layer(max(nx, 64), ny=ny)
    p.s, p.Pr = np.zeros(16), 1.0
    rng = np.random.default_rng(nx + ny)
    saw = 0.25 * (-1.0) ** (np.arange(nx)[None, :] + np.arange(ny)[:, None])
    base = np.concatenate([np.full(4, 8.0), rng.uniform(0.5, 2.0, 12)])
    f = base[:, None, None] * (1.0 + saw * (1.0 + eps * rng.uniform(-1.0, 1.0, (16, ny, nx))))
    want = _step(lbm, p, 1, f)
    got = _step(lbm, p, kernel, f)
    assert np.abs(got - want).max() <= 16 * 2.0 ** -47 * np.abs(f).max()


@pytest.mark.parametrize("kernel", [8, 9])
def test_a_nan_stays_within_one_cell_of_a_step(lbm, kernel):
    """The slope of a cell next to a NaN is zero (its differences do not agree in sign): a step
    carries a NaN one cell along its motion and no further, as in the float64 kernels."""
    p = wl.shear_layer(64, ny=48)
    p.s, p.Pr = np.zeros(16), 1.0
    rng = np.random.default_rng(3)
    f = 1.0 + 0.1 * rng.uniform(-1.0, 1.0, (16, 48, 64))
    f[:, 20, 30] = np.nan
    bad = ~np.isfinite(_step(lbm, p, kernel, f))
    y, x = np.nonzero(bad.any(axis=0))
    assert bad[:, 20, 30].all() and abs(y - 20).max() <= 1 and abs(x - 30).max() <= 1
    assert np.array_equal(bad, ~np.isfinite(_step(lbm, p, 1, f)))
