"""The complex128 sweeps, which run in 64-bit fixed point with one scale per line.

Tolerances.  A line is held to at least 50 bits below its rms value and picks up
a few roundings of that size per step; 20 steps stay below 20 * 16 * 2^-50 =
2.8e-13 in relative L2 whatever the line length.  Angles of up to 100 rad carry
a relative 2^-52 each, 2.2e-14, times a few factors: 1e-12.
"""
import math

import numpy as np
import pytest

import gpe_inputs as gi

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gpe():
    import torch
    import paper_2301_08275_gb300 as g
    g.build()
    g.lib()
    assert torch.cuda.is_available()
    return g


def rel(a, b):
    return float(np.linalg.norm(np.ravel(a) - np.ravel(b)) / np.linalg.norm(np.ravel(b)))


def spec(n, g=30.0, dt=1e-3, gamma=1.0):
    d = len(n)
    L = [12.0, 10.0, 8.0][:d]
    return gi.Spec(n=n, lo=tuple(-x / 2 for x in L), length=tuple(L), g=g, dt=dt, gamma=(gamma, 1.3 * gamma, 1.7 * gamma)[:d])


def run(gpe, sp, psi0, steps, imag=False, V=None):
    import torch
    p = gpe.Plan(sp.n, sp.lo, sp.length, g=sp.g, dt=sp.dt, gamma=None if V is not None else sp.gamma[: sp.ndim],
                 prec=gpe.GPE_C128, V=V)
    x = torch.from_numpy(np.array(psi0, dtype=np.complex128)).cuda()
    e = None
    if imag:
        _, e = p.step_imag(x, steps, 1.0, 0.0, steps)
    else:
        p.step_real(x, steps)
    torch.cuda.synchronize()
    out = x.cpu().numpy()
    p.close()
    return (out, e) if imag else out


# one-pass lines, every radix remainder, the longest lines, partly filled tiles
SHAPES = [(2, 2), (4, 8), (2, 4096), (4096, 2), (16, 64), (32, 2048), (1024, 16), (512, 32), (2, 2, 2), (8, 4, 64), (128, 2, 16)]


@pytest.mark.parametrize("imag", [False, True], ids=["real", "imag"])
@pytest.mark.parametrize("n", SHAPES, ids=lambda n: "x".join(map(str, n)))
def test_matches_oracle_at_every_line_length(gpe, orc, n, imag):
    sp = spec(n)
    psi0 = gi.random_field(sp, seed=sum(n), smooth=0.05)
    if imag:
        out, e = run(gpe, sp, psi0, 20, imag=True)
        pr = orc.Problem(**sp.kwargs())
        ref = pr.step_imag(psi0, 20)
        assert abs(e[0] - pr.norm_energy(ref)[4]) <= 1e-12 * abs(e[0])
    else:
        out = run(gpe, sp, psi0, 20)
        ref = orc.Problem(**sp.kwargs()).step_real(psi0, 20)
    assert rel(out, ref) < 2.8e-13


@pytest.mark.parametrize("g,dt,gamma", [(-20.0, 1e-3, 1.0), (2000.0, 0.02, 1.0), (0.0, -1e-3, 1.0)])
def test_angles_of_every_size(gpe, orc, g, dt, gamma):
    """Small angles, angles past 1/64 turn, past a turn, of either sign, and backwards in time."""
    sp = spec((64, 32), g=g, dt=dt, gamma=gamma)
    psi0 = gi.harmonic_gaussian(sp, seed=1, noise=0.05)
    assert rel(run(gpe, sp, psi0, 1), orc.Problem(**sp.kwargs()).step_real(psi0, 1)) < 1e-12


@pytest.mark.parametrize("imag", [False, True], ids=["real", "imag"])
def test_large_sampled_potential(gpe, orc, imag):
    sp = spec((32, 64), dt=0.01, gamma=0.0)
    V = np.random.default_rng(3).uniform(0, 2000 if not imag else 400, size=sp.shape)
    psi0 = gi.random_field(sp, seed=4, smooth=0.05)
    pr = orc.Problem(**sp.kwargs(), V=V)
    out = run(gpe, sp, psi0, 1, imag=imag, V=V)
    assert rel(out[0] if imag else out, (pr.step_imag if imag else pr.step_real)(psi0, 1)) < 1e-12


def test_scale_is_per_line_and_exact(gpe):
    """Without interaction a step is linear: scaling the state by a power of two
    scales the result by it, bit for bit, down to lines of very small values."""
    sp = spec((64, 128), g=0.0)
    psi0 = gi.random_field(sp, seed=9, smooth=0.02)
    out = run(gpe, sp, psi0, 3)
    for s in (2.0 ** 300, 2.0 ** -300):
        assert np.array_equal(run(gpe, sp, psi0 * s, 3), out * s)
    assert not np.any(run(gpe, sp, np.zeros_like(psi0), 3))


@pytest.mark.parametrize("bad", [np.nan, np.inf, complex(0, -np.inf)])
def test_non_finite_values_spread(gpe, bad):
    sp = spec((64, 32), g=0.0)
    psi0 = gi.random_field(sp, seed=2)
    psi0[7, 5] = bad
    assert np.isnan(run(gpe, sp, psi0, 1)).all()
    import torch
    x = torch.from_numpy(psi0).cuda()
    p = gpe.Plan(sp.n, sp.lo, sp.length, g=sp.g, dt=sp.dt, gamma=sp.gamma[:2], prec=gpe.GPE_C128)
    with pytest.raises(gpe.GpeError):
        p.step_imag(x, 4, 1.0, 0.0, 2)
    p.close()


def test_norm_over_many_steps(gpe):
    """Unit factors of 62 bits and integer sums: no drift beyond a random walk of
    one 2^-53 rounding per point and pass."""
    sp = spec((128, 64), g=50.0)
    psi0 = gi.harmonic_gaussian(sp, seed=1, noise=0.05)
    n0 = math.fsum(np.ravel(np.abs(psi0) ** 2))
    n1 = math.fsum(np.ravel(np.abs(run(gpe, sp, psi0, 2000)) ** 2))
    assert abs(n1 / n0 - 1) < 2e-14
