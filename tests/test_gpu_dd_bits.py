"""The double-float float64 kernels round as their scalar form does, operation for operation.

A product of two double-float numbers adds its two cross terms one after the other, so the order of its
operands is part of the result.  With dy = 1.25 dx the weights of the energy-flux correction have low
parts, and an exchanged pair of operands shows.  The digests are those of the scalar form (one population at
a time, 32 x 32 tiles) on inputs that are exact binary fractions; they hold for the coefficients as an aarch64
host forms them.
"""
import hashlib
import platform

import numpy as np
import pytest

from paper_1305_4736_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

DIGESTS = {0: "03759632726adc74", 1: "a02a53bb71baf1a6", 2: "fddb0a5273a788ef"}


@pytest.fixture(scope="module")
def lbm():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_1305_4736_gb300 import build, lbm as L
    build.build()
    L.load()
    return L


def digest(lbm, limiter, kernel, steps=10, nx=320, ny=160):
    p = wl.shear_layer(512, ny=ny)
    p.nx, p.limiter, p.dy = nx, limiter, 1.25 * p.dx
    # populations near a moving equilibrium, multiples of 2^-30 from an integer recurrence
    k = np.arange(16 * ny * nx, dtype=np.uint64)
    noise = ((k * np.uint64(2862933555777941757) + np.uint64(3037000493)) >> np.uint64(40)).astype(np.float64) * 2.0 ** -30
    base = np.repeat([0.11, 0.0026, 0.17, -0.045], 4)
    f = np.round(base * 2.0 ** 20)[:, None, None] * 2.0 ** -20 * np.ones((16, ny, nx)) + noise.reshape(16, ny, nx)
    s = lbm.Solver.from_problem(p, step_kernel=kernel)
    s.set_state(f)
    s.step(steps)
    out = s.get_state()
    s.close()
    assert np.isfinite(out).all()
    return hashlib.sha256(out.tobytes()).hexdigest()[:16]


@pytest.mark.parametrize("limiter", [0, 1, 2])
@pytest.mark.parametrize("kernel", [8, 9])
def test_bits_of_the_scalar_form(lbm, limiter, kernel):
    if platform.machine() != "aarch64":
        pytest.skip("digests recorded with the coefficients of an aarch64 host")
    assert digest(lbm, limiter, kernel) == DIGESTS[limiter]
