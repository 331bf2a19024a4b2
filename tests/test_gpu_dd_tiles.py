"""Tile edges and the population split of the double-float float64 kernels.

The wide tiles hold 32 x 16 cells, two rows per thread; the narrow ones 32 x 4.  Grids one row or
column either side of a multiple of the tile, every limiter, with and without the energy-flux
correction, are compared with the float64 tile kernel (step_kernel 2) and the two shapes with each
other.  Each double-float operation rounds at about 2^-47 = 7e-15; 20 steps of some hundred
operations on values of at most the largest population stay below 1e-12 of it.
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


def _state(lbm, p, kernel, steps, state=None):
    s = lbm.Solver.from_problem(p, step_kernel=kernel)
    if state is None:
        s.init(*p.fields())
    else:
        s.set_state(state)
    s.step(steps)
    f = s.get_state()
    s.close()
    return f


@pytest.mark.parametrize("limiter", [0, 1, 2])
@pytest.mark.parametrize("nx,ny", [(32, 32), (33, 33), (63, 47), (64, 48), (65, 49), (97, 35)])
def test_wide_and_narrow_tiles_against_the_float64_kernel(lbm, nx, ny, limiter):
    p = wl.shear_layer(nx, ny=ny, seed=nx + ny)
    p.bc = [(wl.BC_NEQ_WALL, 1.0, 0.0, 0.02, 1.01), (wl.BC_ZERO_GRADIENT, 0, 0, 0, 0),
            (wl.BC_EQUILIBRIUM, 1.02, 0.01, 0.0, 1.0), (wl.BC_NEQ_WALL, 1.0, 0.05, 0.0, 1.0)]
    p.limiter = limiter
    p.s = p.s if (nx + limiter) % 2 else wl.rates(5e4)        # Pr = 0.71 or 1 (no energy-flux correction)
    p.Pr = float(p.s[7] / p.s[4])
    want = _state(lbm, p, 2, 20)
    wide = _state(lbm, p, 8, 20)
    assert np.abs(wide - want).max() <= 1e-12 * np.abs(want).max()
    assert np.array_equal(wide, _state(lbm, p, 9, 20))


@pytest.mark.parametrize("seed", range(6))
@pytest.mark.parametrize("kernel", [8, 9])
def test_split_and_rounding_of_populations(lbm, kernel, seed):
    """A uniform state with every rate 0 neither relaxes nor convects: a step returns each
    population through the split and the rounding alone.  The split keeps hi (24 bits, rounded) and
    the remainder (at most 2^-25 of the value) to 24 bits: the result is within 2^-49 of the
    population, exact where 48 bits hold it, and zero below the flush threshold 2^-74."""
    p = wl.shear_layer(40, ny=36)
    p.s, p.Pr = np.zeros(16), 1.0
    rng = np.random.default_rng(seed)
    v = rng.uniform(0.5, 2.0, 16) * 2.0 ** rng.integers(-70, 3, 16) * rng.choice([-1.0, 1.0], 16)
    v[0] = 40.0                                              # the density stays positive
    v[3:6] = (0.0, 1e-30, -(2.0 ** -75))
    v[6:12] = (2.0 ** -74, 1.0 + 2.0 ** -24, -(1.0 + 3 * 2.0 ** -24), 0.5 - 2.0 ** -25, 2.0 - 2.0 ** -24, 1.0 + 2.0 ** -47)
    f = np.broadcast_to(v[:, None, None], (16, p.ny, p.nx))
    got = _state(lbm, p, kernel, 1, np.ascontiguousarray(f))
    assert (got == got[:, :1, :1]).all()
    g = got[:, 0, 0]
    assert (g[3:6] == 0.0).all() and np.array_equal(g[6:12], v[6:12])
    assert (np.abs(g - v)[6:] <= 2.0 ** -49 * np.abs(v)[6:]).all() and (np.abs(g - v)[:3] <= 2.0 ** -49 * np.abs(v)[:3]).all()
