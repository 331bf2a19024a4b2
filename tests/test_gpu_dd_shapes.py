"""The tile shape of the double-float float64 kernels on larger grids.

Kernel 8 takes the shape that was measured fastest (32 x 16 tiles on grids of some waves of them,
32 x 8 on smaller ones); its results on 32 x 16 tiles, whole and ragged, are those of the other shapes bit
for bit and of the plain float64 kernel within 1e-12 of the largest population, the tolerance of the
smaller grids' comparison (each double-float operation rounds at about 2^-47 = 7e-15; 20 steps of some
hundred operations on values of at most the largest population).
"""
import numpy as np
import pytest

from paper_1305_4736_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

WIDE, MID = "DdShape<8, 2, 2", "DdShape<8, 1, 2"
PER, ZG = (wl.BC_PERIODIC, 0, 0, 0, 0), (wl.BC_ZERO_GRADIENT, 0, 0, 0, 0)
MIXED = [(wl.BC_NEQ_WALL, 1.0, 0.0, 0.02, 1.01), ZG, (wl.BC_EQUILIBRIUM, 1.02, 0.01, 0.0, 1.0),
         (wl.BC_NEQ_WALL, 1.0, 0.05, 0.0, 1.0)]
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
    from torch.profiler import ProfilerActivity, profile
    with profile(activities=[ProfilerActivity.CUDA]):        # the first session sets the profiler up
        torch.ones(1, device="cuda").add_(1)
        torch.cuda.synchronize()
    return L


def _solver(lbm, p, kernel):
    s = lbm.Solver.from_problem(p, step_kernel=kernel)
    s.init(*p.fields())
    return s


def _shape_of_a_step(s):
    import torch
    from torch.profiler import ProfilerActivity, profile
    torch.cuda.synchronize()
    with profile(activities=[ProfilerActivity.CUDA]) as prof:
        s.step(1)
        torch.cuda.synchronize()
    names = [e.name for e in prof.events() if "k_step_dd" in e.name]
    return names[0] if names else None


@pytest.mark.parametrize("nx,ny,shape", [(256, 256, MID), (380, 380, MID), (400, 400, MID), (608, 512, WIDE),
                                         (1023, 517, WIDE), (1000, 700, WIDE)])
def test_kernel_8_takes_the_faster_shape(lbm, nx, ny, shape):
    import torch
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("measured on 152 SMs")
    s = _solver(lbm, wl.shear_layer(nx, ny=ny), 8)
    name = _shape_of_a_step(s)
    s.close()
    if name is None:
        pytest.skip("the profiler records no launches here")
    assert shape in name


@pytest.mark.parametrize("edges", ["mixed", "walls", "periodic"])
@pytest.mark.parametrize("limiter", [0, 1, 2])
@pytest.mark.parametrize("nx,ny", [(1023, 517), (1000, 700)])
def test_wide_tiles_against_the_other_kernels(lbm, nx, ny, limiter, edges):
    p = wl.shear_layer(nx, ny=ny, seed=nx + ny)
    p.bc = {"mixed": MIXED, "walls": WALLS, "periodic": [PER] * 4}[edges]
    p.limiter = limiter
    p.s = p.s if (nx + limiter) % 2 else wl.rates(5e4)        # Pr = 0.71 or 1 (no energy-flux correction)
    p.Pr = float(p.s[7] / p.s[4])
    out = {}
    for kernel in (1, 8, 9):
        s = _solver(lbm, p, kernel)
        s.step(20)
        out[kernel] = s.get_state()
        s.close()
    assert np.abs(out[8] - out[1]).max() <= 1e-12 * np.abs(out[1]).max()
    assert np.array_equal(out[8], out[9])
