"""Imaginary-time factors of any size in complex128: exponents far beyond those of a
ground-state run, and kinetic factors beyond the range of doubles (dt < 0).

Tolerance: a factor exp(-x) from a double x carries x 2^-53 (x up to 290 per
half-step here: 3.2e-14), two half-steps a step, two steps, on both sides: 2.6e-13;
rounded up to 1e-12.
"""
import numpy as np
import pytest

import gpe_inputs as gi

pytestmark = pytest.mark.gpu

# (64, 64) is stepped on chip, the others by sweeps
SHAPES = [(64, 64), (32, 64), (16, 8, 16)]


@pytest.fixture(scope="module")
def gpe():
    import torch
    import paper_2301_08275_gb300 as g
    g.build()
    g.lib()
    assert torch.cuda.is_available()
    return g


def step(gpe, sp, psi0, steps, V=None):
    import torch
    p = gpe.Plan(sp.n, sp.lo, sp.length, g=sp.g, dt=sp.dt, gamma=None if V is not None else sp.gamma[: sp.ndim],
                 prec=gpe.GPE_C128, V=V)
    x = torch.from_numpy(np.array(psi0, dtype=np.complex128)).cuda()
    try:
        p.step_imag(x, steps, 1.0, 0.0, steps)
    finally:
        p.close()
    return x.cpu().numpy()


def rel(a, b):
    return float(np.linalg.norm(np.ravel(a) - np.ravel(b)) / np.linalg.norm(np.ravel(b)))


@pytest.mark.parametrize("x0", [20.0, 23.0, 25.0])
@pytest.mark.parametrize("n", SHAPES, ids=lambda n: "x".join(map(str, n)))
def test_box_far_up_the_trap(gpe, orc, n, x0):
    """V dt / 2 of 100 to 180 on one axis, growing by some 30 across the box."""
    d = len(n)
    sp = gi.Spec(n=n, lo=(x0,) + (-1.0,) * (d - 1), length=(2.0,) * d, g=5.0, dt=1.0, gamma=(1.0, 0.7, 0.4)[:d])
    psi0 = gi.random_field(sp, seed=3, smooth=0.05)
    assert rel(step(gpe, sp, psi0, 2), orc.Problem(**sp.kwargs()).step_imag(psi0, 2)) < 1e-12


@pytest.mark.parametrize("n", SHAPES, ids=lambda n: "x".join(map(str, n)))
def test_high_sampled_potential(gpe, orc, n):
    d = len(n)
    sp = gi.Spec(n=n, lo=(-1.0,) * d, length=(2.0,) * d, g=5.0, dt=1.0, gamma=(0.0,) * d)
    V = np.random.default_rng(5).uniform(300.0, 340.0, size=sp.shape)       # V dt / 2 log2(e) of 216 to 245
    psi0 = gi.random_field(sp, seed=4, smooth=0.05)
    assert rel(step(gpe, sp, psi0, 2, V=V), orc.Problem(**sp.kwargs(), V=V).step_imag(psi0, 2)) < 1e-12


@pytest.mark.parametrize("n", [(64, 64), (32, 64), (8, 8, 64)], ids=lambda n: "x".join(map(str, n)))
def test_kinetic_factor_beyond_doubles_is_reported(gpe, n):
    """dt < 0: exp(k^2 |dt| / 2) overflows on the last axis alone."""
    d = len(n)
    sp = gi.Spec(n=n, lo=(-6.0,) * d, length=(60.0,) * (d - 1) + (5.0,), g=0.0, dt=-1.0, gamma=(0.0,) * d)
    with pytest.raises(gpe.GpeError) as ei:
        step(gpe, sp, gi.random_field(sp, seed=1, smooth=0.05), 2)
    assert ei.value.status == 5
