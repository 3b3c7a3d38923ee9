"""A line or an instance gives the same bits alone and in company: the number of
instances of a plan chooses kernels, CTAs and tiles, never a line's arithmetic."""
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


@pytest.mark.parametrize("imag", [False, True], ids=["real", "imag"])
@pytest.mark.parametrize("prec", [0, 1], ids=["c64", "c128"])
@pytest.mark.parametrize("n", [8, 32, 64, 128, 256, 512, 1024, 2048, 4096])
def test_lines_alone_and_in_company(gpe, n, prec, imag):
    """Below and above two lines per SM, one CTA per line (complex128 real time has a
    cluster kernel for up to 32 lines, switched off here: it factors differently)."""
    import torch
    sp = gi.Spec(n=(n,), lo=(-6.0,), length=(12.0,), g=20.0, dt=1e-3, gamma=(1.0,))
    few = np.stack([gi.random_field(sp, seed=b, smooth=0.05) for b in range(3)])
    dt = torch.complex128 if prec else torch.complex64
    out = []
    for batch in (3, 700):
        p = gpe.Plan(sp.n, sp.lo, sp.length, g=sp.g, dt=sp.dt, gamma=sp.gamma[:1], prec=prec, batch=batch,
                     g_each=[sp.g + b % 3 for b in range(batch)])
        p.set_option(gpe.GPE_OPT_LINE_CLUSTER, 0)
        x = torch.from_numpy(few[np.arange(batch) % 3]).cuda().to(dt)
        if imag:
            p.step_imag(x, 5, 1.0, 0.0, 5)
        else:
            p.step_real(x, 5)
        torch.cuda.synchronize()
        out.append(x.cpu().numpy())
        p.close()
    for b in (0, 1, 2, 303, 304, 698, 699):
        assert np.array_equal(out[1][b], out[0][b % 3]), b


def imag(gpe, sp, psi, prec, batch, steps, option=None, V=None):
    import torch
    p = gpe.Plan(sp.n, sp.lo, sp.length, g=sp.g, dt=sp.dt, gamma=None if V is not None else sp.gamma[:2], prec=prec,
                 batch=batch, g_each=[sp.g + b % 3 for b in range(batch)], V=V)
    if option is not None:
        p.set_option(option, 0)
    x = torch.from_numpy(psi[np.arange(batch) % 3]).cuda().to(torch.complex128 if prec else torch.complex64)
    p.trace()
    p.step_imag(x, steps, 1.0, 0.0, steps)
    torch.cuda.synchronize()
    kinds = p.trace_read()
    p.close()
    return x.cpu().numpy(), {k.split(":")[0] for k in kinds if not k.endswith("diag")}


@pytest.mark.parametrize("prec", [0, 1], ids=["c64", "c128"])
@pytest.mark.parametrize("sampled", [False, True], ids=["trap", "sampled"])
@pytest.mark.parametrize("n", [(64, 64), (64, 128), (128, 64), (128, 128)], ids=lambda n: "x".join(map(str, n)))
def test_imaginary_time_on_chip_and_as_sweeps(gpe, n, sampled, prec):
    """2D grids of 64 or 128 points per axis are stepped on chip up to 2^17 points in
    all, as sweeps beyond and with an option of the sweeps: the same bits."""
    sp = gi.Spec(n=n, lo=(-6.0, -5.0), length=(12.0, 10.0), g=50.0, dt=1e-3, gamma=(0.0, 0.0) if sampled else (1.0, 1.4))
    V = gi.anharmonic(sp, gamma=(1.0, 1.5), lam=0.1) if sampled else None
    psi = np.stack([gi.random_field(sp, seed=b, smooth=0.03) for b in range(3)])
    most = (1 << 17) // (n[0] * n[1])
    a, ka = imag(gpe, sp, psi, prec, 3, 12, V=V)
    b, kb = imag(gpe, sp, psi, prec, 3, 12, gpe.GPE_OPT_TILE_X, V=V)
    at, kat = imag(gpe, sp, psi, prec, most, 12, V=V)
    over, kover = imag(gpe, sp, psi, prec, most + 1, 12, V=V)
    plane = {"plane%dx%d" % n}
    assert ka == kat == plane and kb == kover == {"x%d" % n[0], "y%d" % n[1]}
    assert np.array_equal(a, b)
    for i in range(most + 1):
        assert np.array_equal(over[i], a[i % 3]), i
        assert i == most or np.array_equal(at[i], a[i % 3]), i


@pytest.mark.parametrize("prec", [0, 1], ids=["c64", "c128"])
@pytest.mark.parametrize("n", [(8, 256, 256), (128, 64, 64), (128, 16, 128)], ids=lambda n: "x".join(map(str, n)))
def test_sums_of_several_instances_of_several_chunks(gpe, n, prec):
    """More than 4096 lines per instance and axis: chunk sums, added per instance."""
    import torch
    sp = gi.Spec(n=n, lo=(-6.0,) * 3, length=(12.0,) * 3, g=20.0, dt=1e-3, gamma=(1.0, 1.2, 1.4))
    psi = np.stack([(1 + b) * gi.random_field(sp, seed=b, smooth=0.05) for b in range(5)])
    psi = torch.from_numpy(psi).cuda().to(torch.complex128 if prec else torch.complex64)

    def values(x, g):
        p = gpe.Plan(sp.n, sp.lo, sp.length, g=0.0, dt=sp.dt, gamma=sp.gamma, prec=prec, batch=len(g), g_each=g)
        x = x.clone()
        out = [p.norm_energy(x), p.rms_size(x), p.norm_energy(x)]
        _, e = p.step_imag(x, 3, 1.0, 0.0, 1)
        torch.cuda.synchronize()
        p.close()
        return out + [np.reshape(e, -1), x.cpu().numpy()]

    g = [5.0 * b for b in range(5)]
    many = values(psi, g)
    for b in range(5):
        for m, one in zip(many, values(psi[b:b + 1], g[b:b + 1])):
            assert np.array_equal(m[b], one[0])


def planes(count, seed):
    """2D instances that are stepped on chip when grouped, each with its own g and trap."""
    rng = np.random.default_rng(seed)
    shapes = [(128, 64), (64, 128), (128, 128), (64, 64)]
    return [gi.Spec(n=shapes[i % 4], lo=(-6.0, -6.0), length=(12.0, 12.0), g=float(rng.uniform(0, 200)), dt=1e-3,
                    gamma=tuple(float(v) for v in rng.uniform(1.0, 3.0, size=2))) for i in range(count)]


def as_sweeps(gpe, sp, psi, prec, imag, nsteps, check_every=1):
    import torch
    p = gpe.Plan(sp.n, sp.lo, sp.length, g=sp.g, dt=sp.dt, gamma=sp.gamma[:2], prec=prec)
    p.set_option(gpe.GPE_OPT_TILE_X, 0)
    x = torch.from_numpy(psi.copy()).cuda()
    if imag:
        p.step_imag(x, nsteps, 1.0, 0.0, check_every)
    else:
        p.step_real(x, nsteps)
    torch.cuda.synchronize()
    p.close()
    return x.cpu().numpy()


@pytest.mark.parametrize("prec", [0, 1], ids=["c64", "c128"])
def test_planes_of_a_batch_keep_their_parameters(gpe, prec):
    import torch
    dt = np.complex128 if prec else np.complex64
    specs = planes(16, seed=prec)
    psi = [gi.random_field(sp, seed=i, smooth=0.05).astype(dt) for i, sp in enumerate(specs)]
    xs = [torch.from_numpy(p.copy()).cuda() for p in psi]
    descs = [gpe.make_desc(sp.n, sp.lo, sp.length, g=sp.g, dt=sp.dt, gamma=sp.gamma[:2], prec=prec)[0] for sp in specs]
    b = gpe.gpe_batch_create(descs, torch.cuda.current_stream().cuda_stream)
    gpe.gpe_batch_step_real(b, [x.data_ptr() for x in xs], 9, True)
    torch.cuda.synchronize()
    gpe.gpe_batch_destroy(b)
    for i, sp in enumerate(specs):
        assert np.array_equal(xs[i].cpu().numpy(), as_sweeps(gpe, sp, psi[i], prec, False, 9)), i


@pytest.mark.parametrize("prec", [0, 1], ids=["c64", "c128"])
def test_planes_of_a_server_keep_their_slots(gpe, prec):
    """More requests than places, of different lengths: slots are handed on, and the
    members of a round are not in the order of their slots."""
    dt = np.complex128 if prec else np.complex64
    specs = [sp for sp in planes(40, seed=10 + prec) if sp.n in ((128, 64), (64, 64))]
    psi = [gi.random_field(sp, seed=i, smooth=0.05).astype(dt) for i, sp in enumerate(specs)]
    nsteps = [5 * (1 + (7 * i) % 11) for i in range(len(specs))]
    srv = gpe.gpe_server_create(1 << 30, max_active=7, chunk_steps=5)
    tickets = [gpe.gpe_serve_submit(srv, gpe.make_desc(sp.n, sp.lo, sp.length, g=sp.g, dt=sp.dt, gamma=sp.gamma[:2],
                                                       prec=prec)[0], psi[i], imag=i % 3 > 0, nsteps=nsteps[i],
                                    etol=0.0, check_every=5) for i, sp in enumerate(specs)]
    for i, t in enumerate(tickets):
        out = np.empty_like(psi[i])
        r = gpe.gpe_serve_poll(srv, t, timeout_ms=-1, psi_out=out)
        assert r.status == 0 and r.steps_done == nsteps[i]
        if i % 3 > 0:
            assert np.array_equal(out, as_sweeps(gpe, specs[i], psi[i], prec, True, nsteps[i], 5)), i
        else:      # real-time requests advance in chunks; a chunk ends and opens the nonlinear half-step
            assert np.linalg.norm(out - as_sweeps(gpe, specs[i], psi[i], prec, False, nsteps[i])) < \
                (1e-12 if prec else 1e-4) * np.linalg.norm(out), i
    gpe.gpe_server_destroy(srv)
