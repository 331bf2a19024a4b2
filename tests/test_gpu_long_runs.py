"""Graphs of 16 steps (calls of 64 steps or more) and the own launches of large batch members, bit for
bit against the same steps one a call.  (A member on the plain kernel shares the packed plain kernel, whose
multiply-add contraction may differ: to round-off, as in test_gpu_batch.py.)"""
import numpy as np
import pytest

from paper_1305_4736_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

WALLS = [(wl.BC_NEQ_WALL, 1.0, 0.0, 0.02, 1.01), (wl.BC_NEQ_WALL, 1.0, 0.0, -0.03, 0.99),
         (wl.BC_NEQ_WALL, 1.0, 0.02, 0.0, 1.0), (wl.BC_NEQ_WALL, 1.0, 0.05, 0.0, 1.0)]


@pytest.fixture(scope="module")
def lbm():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_1305_4736_gb300 import build, lbm as L
    build.build()
    L.load()
    return L


def _shear(nx, ny, walls=False, limiter=0, seed=7):
    p = wl.shear_layer(max(nx, 64), ny=ny, seed=seed)
    p.nx = nx
    p.rho, p.ux, p.uy, p.T = (np.ascontiguousarray(a[:, :nx]) for a in p.fields())
    if walls:
        p.bc = WALLS
    p.limiter = limiter
    return p


def _solver(lbm, p, precision, kernel=0):
    s = lbm.Solver.from_problem(p, precision=precision, step_kernel=kernel)
    s.init(*p.fields())
    return s


CASES = [(200, 4, False, 0, 9), (200, 4, False, 1, 1), (256, 256, True, 0, 9), (512, 320, False, 0, 8),
         (256, 128, True, 1, 2), (4, 200, True, 0, 7), (40, 300, True, 0, 3), (300, 200, True, 1, 4),
         (256, 64, False, 0, 5), (256, 64, True, 1, 6)]


@pytest.mark.parametrize("nx,ny,walls,precision,kernel", CASES)
def test_long_calls_equal_single_steps(lbm, nx, ny, walls, precision, kernel):
    p = _shear(nx, ny, walls)
    a, b = _solver(lbm, p, precision, kernel), _solver(lbm, p, precision, kernel)
    for n in (1, 64, 81, 17, 96):                 # 16-step graphs from either buffer, with steps left over
        a.step(n)
    for _ in range(259):
        b.step(1)
    assert a.step_count == b.step_count == 259
    assert np.array_equal(a.get_state(), b.get_state())
    a.close()
    b.close()


def test_long_call_after_autotune(lbm):
    p = _shear(512, 320)
    a = _solver(lbm, p, 0)
    a.step(80)
    choice = a.autotune(2)
    b = lbm.Solver.from_problem(p, step_kernel=choice)
    b.set_state(a.get_state())
    a.step(65)
    for _ in range(65):
        b.step(1)
    assert np.array_equal(a.get_state(), b.get_state())


BATCHES = {
    # one launch a step: chained, in graphs of 16 steps
    "float32 tiles": [(96, 40, False, 1, 0), (100, 70, False, 1, 0), (333, 129, False, 1, 0)],
    "float64 tiles": [(96, 40, True, 0, 0), (100, 70, False, 0, 0), (161, 97, True, 0, 0)],
    # large members with launches of their own, beside each other and small ones
    "float32 large": [(640, 512, False, 1, 0), (700, 500, True, 1, 0), (1000, 300, False, 1, 0)],
    "float32 large and small": [(640, 512, True, 1, 0), (700, 500, False, 1, 0), (96, 40, False, 1, 0)],
    "float32 small mean": [(640, 512, False, 1, 0), (96, 40, False, 1, 0), (64, 48, False, 1, 0)],
    "float64 large": [(640, 250, False, 0, 0), (700, 269, True, 0, 0), (1000, 332, False, 0, 0)],
    "float64 large and small": [(1023, 517, True, 0, 0), (700, 269, False, 0, 0), (100, 13, True, 0, 0)],
    "float64 small mean": [(640, 250, False, 0, 0), (100, 70, True, 0, 0), (64, 48, False, 0, 0)],
    # both precisions, limiters, a streaming and a plain float32 member
    "mixed": [(640, 512, True, 1, 0), (700, 269, True, 0, 1), (1280, 1024, False, 0, 0), (700, 500, False, 1, 2),
              (300, 100, True, 0, 0), (20, 90, True, 1, 0)],
}


@pytest.mark.parametrize("name", sorted(BATCHES))
def test_batches_equal_stepping_alone(lbm, name):
    specs = BATCHES[name]
    probs = [_shear(nx, ny, walls, limiter, seed=11 + k) for k, (nx, ny, walls, _, limiter) in enumerate(specs)]
    batched = [_solver(lbm, p, spec[3]) for p, spec in zip(probs, specs)]
    alone = [_solver(lbm, p, spec[3]) for p, spec in zip(probs, specs)]
    b = lbm.Batch(batched)
    for n in (65, 1, 4):                          # 16-step graphs where there is one launch, pairs, direct steps
        b.step(n)
    batched[0].step(1)
    alone[0].step(1)
    b.step(67)
    for s in alone:
        for n in (64, 73):
            s.step(n)
    for k, (x, y) in enumerate(zip(batched, alone)):
        assert x.step_count == y.step_count
        got, want = x.get_state(), y.get_state()
        if y.step_kernel == 1:                    # the packed plain kernel: the same to float32 round-off
            assert np.abs(got - want).max() <= 2e-5 * np.abs(want).max(), (name, specs[k])
        else:
            assert np.array_equal(got, want), (name, specs[k])
    b.close()
    for s in batched + alone:
        s.close()
