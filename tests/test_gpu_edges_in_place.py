"""Boundaries read in place by the step kernels.

The tile kernels fill periodic and zero-gradient ghost cells in their staged tile and the plain
kernels read those cells' sources directly; only the streaming kernel (step_kernel 5) still steps on
a full ghost fill.  Each of them is compared with it over the boundary kinds, on grids whose last
tiles are ragged in both directions, alone and in a batch.  Tolerances are those of the kernels'
comparisons elsewhere: 1e-12 of the largest population in float64 (double-float arithmetic), 2e-5 of
it in the float32 mode.
"""
import numpy as np
import pytest

from paper_1305_4736_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

PER, ZG = (wl.BC_PERIODIC, 0, 0, 0, 0), (wl.BC_ZERO_GRADIENT, 0, 0, 0, 0)
EQ = (wl.BC_EQUILIBRIUM, 1.02, 0.03, 0.01, 1.01)
WALL = (wl.BC_NEQ_WALL, 1.0, 0.02, 0.0, 1.01)
EDGES = {"periodic": [PER] * 4, "zero_gradient": [ZG] * 4, "equilibrium": [EQ] * 4, "inflow_outflow": [EQ, ZG, PER, PER],
         "channel": [PER, PER, WALL, WALL], "mixed": [ZG, EQ, WALL, ZG], "walls": [WALL] * 4}


@pytest.fixture(scope="module")
def lbm():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_1305_4736_gb300 import build, lbm as L
    build.build()
    L.load()
    return L


def _problem(edges, nx, ny):
    p = wl.shear_layer(nx, ny=ny, seed=nx + ny)
    p.ux = p.ux + 0.03 * np.sin(2 * np.pi * (np.arange(nx) + 0.5) / nx)[None, :]     # every edge sees a flow
    p.uy = p.uy + 0.02 * np.cos(2 * np.pi * (np.arange(ny) + 0.5) / ny)[:, None]
    p.bc = EDGES[edges]
    return p


def _solver(lbm, p, precision, kernel):
    s = lbm.Solver.from_problem(p, precision=precision, step_kernel=kernel)
    s.init(*p.fields())
    return s


def _run(lbm, p, precision, kernel, steps=15):
    s = _solver(lbm, p, precision, kernel)
    s.step(steps)
    f = s.get_state()
    s.close()
    return f


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nx,ny", [(128, 35), (131, 49), (160, 33)])
@pytest.mark.parametrize("edges", sorted(EDGES))
def test_each_kernel_against_the_full_ghost_fill(lbm, edges, nx, ny, precision):
    p = _problem(edges, nx, ny)
    want = _run(lbm, p, precision, 5)
    tol = (2e-5 if precision else 1e-12) * np.abs(want).max()
    for kernel in ((1, 2, 3) if precision else (1, 2, 7, 8, 9)):
        assert np.abs(_run(lbm, p, precision, kernel) - want).max() <= tol, kernel


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("edges", sorted(EDGES))
def test_small_and_narrow_grids_against_the_oracle(orc, lbm, edges, precision):
    """Grids of a few cells: every read is at an edge, periodic reads wrap more than once."""
    for nx, ny in ((1, 1), (2, 3), (5, 40), (40, 2), (33, 5)):
        p = _problem(edges, nx, ny)
        p.dx, p.dt = 1.0 / 64, 1e-5
        got = _run(lbm, p, precision, 0, 10)
        O = orc.Oracle(nx, ny, p.dx, p.dt, p.gamma, p.s, p.limiter, p.bc)
        O.init(*p.fields())
        O.step(10)
        want = O.get_state()
        assert np.abs(got - want).max() <= (2e-5 if precision else 1e-12) * np.abs(want).max(), (nx, ny)


@pytest.mark.parametrize("precision", [0, 1])
def test_batch_of_every_edge_kind_equals_stepping_alone(lbm, precision):
    probs = [_problem(e, nx, ny) for e in sorted(EDGES) for nx, ny in ((131, 49), (40, 5), (4, 40))]
    alone = [_run(lbm, p, precision, 0, 7) for p in probs]
    solvers = [_solver(lbm, p, precision, 0) for p in probs]
    b = lbm.Batch(solvers)
    b.step(7)
    for s, want in zip(solvers, alone):
        assert np.abs(s.get_state() - want).max() <= (2e-5 if precision else 1e-12) * np.abs(want).max()
    b.close()
    for s in solvers:
        s.close()
