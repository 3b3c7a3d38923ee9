"""2D grids of 64 or 128 points per axis, stepped on chip by one cluster per
instance, against the sweeps that other grids take (selected by a tile option).

Real-time steps run the same arithmetic per line: the same bits.  In imaginary
time the norm is summed in another order: relative 2^-53 per step in
complex128 (1e-13 after 12 steps), one unit of the last place of the factor per
step in complex64 (1e-5).
"""
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


def run(gpe, sp, psi0, prec, sweeps, steps, imag=False, batch=1, g_each=None, V=None):
    import torch
    p = gpe.Plan(sp.n, sp.lo, sp.length, g=sp.g, dt=sp.dt, gamma=None if V is not None else sp.gamma[:2], prec=prec,
                 batch=batch, g_each=g_each, V=V)
    if sweeps:
        p.set_option(gpe.GPE_OPT_TILE_X, 0)
    x = torch.from_numpy(psi0.astype(np.complex64 if prec == gpe.GPE_C64 else np.complex128)).cuda()
    done = e = None
    if imag:
        done, e = p.step_imag(x, steps, 1.0, 1e-30, 5)
    else:
        p.step_real(x, steps)
    torch.cuda.synchronize()
    out = x.cpu().numpy()
    p.close()
    return out, done, e


def spec(n, g=50.0):
    return gi.Spec(n=n, lo=(-6.0, -5.0), length=(12.0, 10.0), g=g, dt=1e-3, gamma=(1.0, 1.4))


@pytest.mark.parametrize("steps", [1, 2, 64, 65, 130])
@pytest.mark.parametrize("prec", [0, 1], ids=["c64", "c128"])
@pytest.mark.parametrize("n", [(64, 64), (64, 128), (128, 64), (128, 128)], ids=lambda n: "x".join(map(str, n)))
def test_real_time_gives_the_bits_of_the_sweeps(gpe, orc, n, prec, steps):
    sp = spec(n)
    psi0 = gi.random_field(sp, seed=sum(n) + steps, smooth=0.03)
    a, b = (run(gpe, sp, psi0, prec, s, steps)[0] for s in (False, True))
    assert np.array_equal(a, b)
    if steps == 2:
        ref = orc.Problem(**sp.kwargs()).step_real(psi0, steps)
        assert np.linalg.norm(a - ref) < (1e-12 if prec else 2e-4) * np.linalg.norm(ref)


@pytest.mark.parametrize("prec", [0, 1], ids=["c64", "c128"])
@pytest.mark.parametrize("n", [(64, 64), (128, 64), (64, 128), (128, 128)], ids=lambda n: "x".join(map(str, n)))
def test_imaginary_time_agrees_with_the_sweeps(gpe, n, prec):
    sp = spec(n)
    psi0 = gi.random_field(sp, seed=7, smooth=0.03)
    (a, da, ea), (b, db, eb) = (run(gpe, sp, psi0, prec, s, 12, imag=True) for s in (False, True))
    tol = 1e-13 if prec else 1e-5
    assert da == db == 12
    assert np.linalg.norm(a - b) < tol * np.linalg.norm(b)
    assert abs(ea[0] - eb[0]) < tol * abs(eb[0])


@pytest.mark.parametrize("imag", [False, True], ids=["real", "imag"])
@pytest.mark.parametrize("prec", [0, 1], ids=["c64", "c128"])
def test_instances_and_sampled_potentials(gpe, prec, imag):
    sp = spec((64, 64))
    tol = 0.0 if not imag else 1e-13 if prec else 1e-5
    psi0 = np.stack([gi.random_field(sp, seed=b, smooth=0.03) for b in range(3)])
    a, b = (run(gpe, sp, psi0, prec, s, 6, imag=imag, batch=3, g_each=[0.0, 40.0, -3.0])[0] for s in (False, True))
    assert np.linalg.norm(a - b) <= tol * np.linalg.norm(b)
    sv = gi.Spec(n=sp.n, lo=sp.lo, length=sp.length, g=20.0, dt=1e-3, gamma=(0.0, 0.0))
    V = gi.anharmonic(sv, gamma=(1.0, 1.5), lam=0.1)
    a, b = (run(gpe, sv, psi0[0], prec, s, 6, imag=imag, V=V)[0] for s in (False, True))
    assert np.linalg.norm(a - b) <= tol * np.linalg.norm(b)


@pytest.mark.parametrize("prec", [0, 1], ids=["c64", "c128"])
def test_zero_norm_is_reported(gpe, prec):
    sp = spec((64, 64))
    with pytest.raises(gpe.GpeError) as ei:
        run(gpe, sp, np.zeros(sp.shape, dtype=np.complex128), prec, False, 4, imag=True)
    assert ei.value.status == 5
