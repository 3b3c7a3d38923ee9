"""Shell binning of the spectra on grids and boxes where the shell of a mode is
decided in different ways: cubic boxes (whole numbers), other boxes (single
precision, double next to an edge), rows shorter than a warp, one-point runs.

Tolerances: complex128 1e-12 relative L2 over the shells (rounding of the
transforms); complex64 1e-5, the bound of the other complex64 diagnostics.
"""
import numpy as np
import pytest

import gpe_inputs as gi

pytestmark = pytest.mark.gpu

CASES = [((2, 2), (1.0, 1.0)), ((4, 512), (3.0, 3.0)), ((512, 8), (10.0, 7.0)), ((64, 32), (5.0, 10.0)),
         ((16, 8, 4), (2.0, 2.0, 2.0)), ((8, 32, 16), (6.0, 4.0, 3.0)), ((256, 64), (12.0, 0.37))]


@pytest.fixture(scope="module")
def gpe():
    import torch
    import paper_2301_08275_gb300 as g
    g.build()
    g.lib()
    assert torch.cuda.is_available()
    return g


@pytest.mark.parametrize("scale", [1.0, 1e-12, 1e12])
@pytest.mark.parametrize("prec", ["c128", "c64"])
@pytest.mark.parametrize("n,length", CASES, ids=lambda v: "x".join(str(x) for x in v))
def test_spectra_match_oracle(gpe, orc, n, length, prec, scale):
    import torch
    sp = gi.Spec(n=n, lo=(0.0,) * len(n), length=length, g=1.0, dt=1e-3, gamma=(0.0,) * len(n))
    dt = np.complex128 if prec == "c128" else np.complex64
    psi = (gi.random_field(sp, seed=sum(n)) * scale).astype(dt)
    p = gpe.Plan(n, sp.lo, length, g=1.0, dt=1e-3, prec=gpe.GPE_C128 if prec == "c128" else gpe.GPE_C64)
    kinds = gpe.GPE_SPEC_INC | gpe.GPE_SPEC_COMP | gpe.GPE_SPEC_QP | gpe.GPE_SPEC_NUM
    out = p.spectrum(torch.from_numpy(psi).cuda(), kinds)[:, 0]
    p.close()
    P = orc.Problem(**sp.kwargs())
    ref = list(P.spectrum(psi.astype(np.complex128))) + list(P.spectrum_qp_num(psi.astype(np.complex128)))
    tol = 1e-12 if prec == "c128" else 1e-5
    for got, want in zip(out, ref):
        got = got[: len(want)]
        total = max(np.linalg.norm(want), 1e-3 * np.linalg.norm(ref[0]) + 1e-3 * np.linalg.norm(ref[1]))
        assert np.linalg.norm(got - want) <= tol * total


@pytest.mark.parametrize("n,length", [((64, 128), (9.0, 9.0)), ((256, 64), (10.0, 4.0)), ((64, 128, 64), (5.0, 5.0, 5.0))],
                         ids=lambda v: "x".join(str(x) for x in v))
def test_fused_derivative_and_velocity_sweeps(gpe, orc, n, length):
    """Complex64 grids of at least 64 points per axis form i k psi and the velocity
    inside the transforms' sweeps; the separate kernels (generic passes) give the
    same spectra, to the rounding of single values (1e-6 of the total)."""
    import torch
    sp = gi.Spec(n=n, lo=(0.0,) * len(n), length=length, g=1.0, dt=1e-3, gamma=(0.0,) * len(n))
    psi = gi.random_field(sp, seed=5).astype(np.complex64)
    psi[..., :3] = 0.0                                  # points without density have no velocity
    kinds = gpe.GPE_SPEC_INC | gpe.GPE_SPEC_COMP | gpe.GPE_SPEC_QP
    outs = []
    for generic in (0, 1):
        p = gpe.Plan(n, sp.lo, length, g=1.0, dt=1e-3, prec=gpe.GPE_C64)
        p.set_option(gpe.GPE_OPT_GENERIC_PASSES, generic)
        outs.append(p.spectrum(torch.from_numpy(psi).cuda(), kinds)[:, 0])
        p.close()
    P = orc.Problem(**sp.kwargs())
    ref = list(P.spectrum(psi.astype(np.complex128))) + [P.spectrum_qp_num(psi.astype(np.complex128))[0]]
    for a, b, r in zip(outs[0], outs[1], ref):
        assert np.linalg.norm(a - b) <= 1e-6 * np.linalg.norm(b)
        assert np.linalg.norm(a[: len(r)] - r) <= 1e-5 * np.linalg.norm(r)
