"""Grids with more tile rows than a launch has in its y dimension (65535).

The fields repeat every 32 rows, so every 32 rows of the tall periodic grid evolve as a 32 x 32 grid
does: the state is the small grid's, bit for bit, at the ends, around row 65535 * 16 and in between.
"""
import numpy as np
import pytest

from paper_1305_4736_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

NY = 65535 * 16 + 48              # 32769 times 32 rows


@pytest.fixture(scope="module")
def lbm():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_1305_4736_gb300 import build, lbm as L
    build.build()
    L.load()
    return L


def _problems():
    small = wl.shear_layer(64, ny=32)
    small.nx = 32
    y, x = np.mgrid[0:32, 0:32] * (2.0 * np.pi / 32)
    small.rho, small.T = 1.0 + 0.05 * np.sin(x + y), 1.0 + 0.04 * np.cos(x - 2 * y)
    small.ux, small.uy = 0.05 * np.sin(y), 0.03 * np.cos(x)
    tall = wl.shear_layer(64, ny=32)
    tall.nx, tall.ny = 32, NY
    tall.rho, tall.ux, tall.uy, tall.T = (np.tile(a, (NY // 32, 1)) for a in small.fields())
    return small, tall


def _check(tall, small):
    want = small.get_state()
    for row in (0, 65535 * 8 // 32 * 32, 65535 * 16 // 32 * 32 - 64, NY - 64):
        got = tall.get_state_rows(row, 64)
        assert np.array_equal(got[:, :32], want) and np.array_equal(got[:, 32:], want), row


def test_float64_grid_past_65535_tile_rows(lbm):
    small, tall = _problems()
    s, t = lbm.Solver.from_problem(small, step_kernel=8), lbm.Solver.from_problem(tall)
    assert t.step_kernel == 8
    for a, p in ((s, small), (t, tall)):
        a.init(*p.fields())
        a.step(17)
    _check(t, s)
    t.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_batch_member_past_65535_tile_rows(lbm, precision):
    small, tall = _problems()
    s, t = lbm.Solver.from_problem(small, precision=precision), lbm.Solver.from_problem(tall, precision=precision)
    for a, p in ((s, small), (t, tall)):
        a.init(*p.fields())
    b = lbm.Batch([t])
    b.step(5)
    s.step(5)
    _check(t, s)
    b.close()
    t.close()
