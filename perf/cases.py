"""Timed cases of the TSSP Gross-Pitaevskii library.

Each case is the work that a program hands to the library in one go, through
its public entry points (``Plan``, the batch calls and the request server):
real-time steps, imaginary-time ground states, kinetic-energy spectra and the
norm/energy/size diagnostics, in complex64 and complex128, from a single short
line to a 512^3 grid.  Sizes are those of the workloads in ``gpe_inputs`` and
``bench.py``; grids are powers of two per axis (what the library accepts), so
ragged sizes are unequal axes, thin slabs and uneven batches.

kind      meaning of the fields
"real"    nx, ny, nz (0: axis absent), prec (64 or 128: bits of the complex
          type), batch instances, steps, g, gamma (strength of the harmonic
          trap, 0: none), field ("trap", "vortex", "flow")
"imag"    the same in imaginary time, energies checked every ``every`` steps
"spectra" incompressible and compressible spectra of a field
"energy"  norm/energy/mu and rms sizes of a field
"batch"   count uneven 2D instances of lo^2 ... hi^2 points, steps each
"serve"   count requests of mixed dimension, submitted together and polled
"""
import math

import numpy as np
import torch

import paper_2301_08275_gb300 as gpe

DT = 1e-3


def listed():
    return [
        # the smallest grid of the batched workload on a plan of its own: bound by launches
        dict(name="grid_64_c64", kind="real", nx=64, ny=64, nz=0, prec=64, batch=1, steps=20, g=100.0, gamma=2.0,
             field="trap"),
        # the 1D workload: one 256-point line, 1000 steps in one call
        dict(name="line_256_c128", kind="real", nx=256, ny=0, nz=0, prec=128, batch=1, steps=1000, g=10.0, gamma=1.0,
             field="trap"),
        # the 1D solves of the request stream, a group of them advancing together
        dict(name="lines_4096_c64", kind="real", nx=4096, ny=0, nz=0, prec=64, batch=64, steps=100, g=200.0, gamma=2.0,
             field="trap"),
        # 2D turbulence between two readings of its spectra, both precisions
        dict(name="turbulence_1024_c64", kind="real", nx=1024, ny=1024, nz=0, prec=64, batch=1, steps=100, g=1.0,
             gamma=0.0, field="vortex"),
        dict(name="turbulence_1024_c128", kind="real", nx=1024, ny=1024, nz=0, prec=128, batch=1, steps=20, g=1.0,
             gamma=0.0, field="vortex"),
        # the headline grid: Taylor-Green flow at 512^3
        dict(name="taylor_green_512_c64", kind="real", nx=512, ny=512, nz=512, prec=64, batch=1, steps=6, g=1.0,
             gamma=0.0, field="flow"),
        # 3D trap after the quench, the ten steps between two readings of its size
        dict(name="trap_256_c64", kind="real", nx=256, ny=256, nz=256, prec=64, batch=1, steps=10, g=200.0, gamma=2.0,
             field="trap"),
        # ground states by imaginary time: the bulk of the 3D trap's, and the 2D
        # validation table's in full precision
        dict(name="ground_256_c64", kind="imag", nx=256, ny=256, nz=256, prec=64, batch=1, steps=16, every=16, g=200.0,
             gamma=1.0, field="trap"),
        dict(name="ground_128_c128", kind="imag", nx=128, ny=128, nz=0, prec=128, batch=1, steps=100, every=20,
             g=100.0, gamma=1.0, field="trap"),
        # the spectra that the turbulence run reads
        dict(name="spectra_1024_c64", kind="spectra", nx=1024, ny=1024, nz=0, prec=64, batch=1, g=1.0, gamma=0.0,
             field="vortex"),
        # whole calls: the uneven batch, and a burst of requests to the server
        dict(name="batch_512", kind="batch", count=512, lo=64, hi=512, steps=20),
        dict(name="serve_24", kind="serve", count=24, steps=100),
    ]


# a drawn case stays below these many point-steps (a complex128 point counts
# for sixteen: double precision is slow on this GPU)
_MOST = 6.0e8


def _axis(rng, lo, hi):
    return 1 << rng.randint(int(math.log2(lo)), int(math.log2(hi)))


def draw(rng):
    kind = rng.choices(["real", "imag", "spectra", "energy", "batch", "serve"], [10, 4, 2, 2, 1, 1])[0]
    if kind == "batch":
        lo = _axis(rng, 64, 128)
        return dict(kind=kind, count=rng.randint(16, 400), lo=lo, hi=lo << rng.randint(1, 2), steps=rng.randint(5, 40))
    if kind == "serve":
        return dict(kind=kind, count=rng.randint(6, 24), steps=rng.randint(20, 100))
    prec = rng.choice([64, 64, 128])
    weight = 16 if prec == 128 else 1
    while True:
        d = rng.choice([1, 2, 2, 3, 3]) if kind != "spectra" else rng.choice([2, 3])
        nx = _axis(rng, 64, 4096) if d == 1 else _axis(rng, 32, 2048) if d == 2 else _axis(rng, 32, 512)
        ny = _axis(rng, 32, 2048) if d == 2 else _axis(rng, 32, 512) if d == 3 else 0
        nz = _axis(rng, 32, 512) if d == 3 else 0
        points = nx * max(ny, 1) * max(nz, 1)
        batch = rng.randint(1, 48) if d == 1 else rng.choice([1, 1, 1, rng.randint(2, 9)])
        if kind in ("spectra", "energy"):
            if points * batch * weight <= 1 << 27:
                break
        elif points * batch * weight * 4 <= _MOST:
            break
    case = dict(kind=kind, nx=nx, ny=ny, nz=nz, prec=prec, batch=batch)
    trapped = kind == "imag" or rng.random() < 0.5
    case.update(g=round(rng.uniform(0.0, 400.0), 3) if trapped else 1.0,
                gamma=round(rng.uniform(0.8, 2.0), 3) if trapped else 0.0, field="trap" if trapped else "flow")
    if kind in ("real", "imag"):
        most = max(4, min(1000 if d == 1 else 100, int(_MOST / (points * batch * weight))))
        case["steps"] = int(round(math.exp(rng.uniform(math.log(4), math.log(most)))))
    if kind == "imag":
        case["every"] = rng.choice([5, 10, 20])
    return case


# ------------------------------------------------------------------ inputs
def _shape(case):
    """Points per axis, x first."""
    return tuple(n for n in (case["nx"], case["ny"], case["nz"]) if n)


def _box(case):
    """Corner, length and trap frequencies per axis: a trap that its states fit, or
    a periodic box with the spacing of the turbulence workloads."""
    n = _shape(case)
    if case["gamma"]:
        half = [8.0, 8.0, 6.0][:len(n)]
        gamma = [case["gamma"] * f for f in (1.0, 1.3, 1.7)][:len(n)]
        return [-h for h in half], [2 * h for h in half], gamma
    return [0.0] * len(n), [2 * math.pi * v / 32 for v in n], [0.0] * len(n)


def _coords(n, lo, length, dev):
    """Per-axis coordinates, broadcastable over an array with x fastest."""
    d = len(n)
    out = []
    for a in range(d):
        x = lo[a] + torch.arange(n[a], dtype=torch.float64, device=dev) * (length[a] / n[a])
        out.append(x.reshape([-1 if i == d - 1 - a else 1 for i in range(d)]))
    return out


def _gaussian(n, lo, length, gamma, rng, dev, noise=0.01):
    """Harmonic ground state of the trap, slightly off its centre, with phase noise."""
    amp = torch.ones((), dtype=torch.float64, device=dev)
    for x, ga in zip(_coords(n, lo, length, dev), gamma):
        off = 0.5 * float(rng.uniform(-1, 1))
        amp = amp * ((ga / math.pi) ** 0.25 * torch.exp(-0.5 * ga * (x - off) ** 2))
    gen = torch.Generator(device=dev).manual_seed(int(rng.integers(1 << 31)))
    ph = noise * (2 * torch.rand(amp.shape, generator=gen, dtype=torch.float64, device=dev) - 1)
    return torch.polar(amp.contiguous(), ph)


def _flow(n, lo, length, rng, dev):
    """Taylor-Green phase (in 1D and 2D its cut) with 1 % density noise."""
    x = _coords(n, lo, length, dev)
    k = [4 * 2 * math.pi / v for v in length]
    sh = [float(v) for v in rng.uniform(0, 2 * math.pi, size=len(n))]
    c = [torch.cos(k[a] * x[a] + sh[a]) for a in range(len(n))]
    th = torch.zeros(tuple(reversed(n)), dtype=torch.float64, device=dev)
    for a in range(1, len(n)):
        u, v = torch.broadcast_tensors(c[a], c[0])
        th = th + torch.atan2(u, v)
    if len(n) == 1:
        th = th + 0.5 * c[0]
    gen = torch.Generator(device=dev).manual_seed(int(rng.integers(1 << 31)))
    rho = 1 + 0.01 * (2 * torch.rand(th.shape, generator=gen, dtype=torch.float64, device=dev) - 1)
    return torch.polar(rho.sqrt(), th)


def _vortices(n, length, rng, dev):
    """Alternating point vortices, one per 2048 points, on a periodic box: the phase
    from a product of Jacobi theta functions, the amplitude from tanh cores."""
    nx, ny = n
    nv = max(2, nx * ny // 2048 // 2 * 2)
    (x, y), (lx, ly) = _coords(n, [0.0, 0.0], length, dev), length
    # jittered cells keep the cores apart
    side = int(math.ceil(math.sqrt(nv)))
    cells = rng.permutation(side * side)[:nv]
    px = ((cells % side) + rng.uniform(0.25, 0.75, nv)) * lx / side
    py = ((cells // side) + rng.uniform(0.25, 0.75, nv)) * ly / side
    th = torch.zeros((ny, nx), dtype=torch.float64, device=dev)
    amp = torch.ones((ny, nx), dtype=torch.float64, device=dev)
    q, mom = math.exp(-math.pi * ly / lx), 0.0
    for j in range(nv):
        s = 1.0 if j % 2 == 0 else -1.0
        dx, dy = x - px[j], y - py[j]
        ax, ay = math.pi * dx / lx, math.pi * dy / lx
        re = im = 0.0
        for m in range(3):
            c = 2 * (-1) ** m * q ** ((m + 0.5) ** 2)
            re = re + (c * torch.cosh((2 * m + 1) * ay)) * torch.sin((2 * m + 1) * ax)
            im = im + (c * torch.sinh((2 * m + 1) * ay)) * torch.cos((2 * m + 1) * ax)
        th += s * torch.atan2(im, re)
        rx, ry = dx - lx * torch.round(dx / lx), dy - ly * torch.round(dy / ly)
        amp *= torch.tanh(torch.sqrt(rx ** 2 + ry ** 2).float()).double()
        mom += s * px[j]
    th -= 2 * math.pi * mom * y / (lx * ly)
    return torch.polar(amp, th)


def _field(case, seed):
    """The state of a case: (batch, nz, ny, nx) without the absent axes, on the GPU."""
    dev = torch.device("cuda")
    rng = np.random.default_rng(seed)
    n = _shape(case)
    lo, length, gamma = _box(case)
    dtype = torch.complex64 if case["prec"] == 64 else torch.complex128
    out = torch.empty((case["batch"],) + tuple(reversed(n)), dtype=dtype, device=dev)
    for b in range(case["batch"]):
        if case["field"] == "vortex":
            out[b] = _vortices(n, length, rng, dev)
        elif case["field"] == "flow":
            out[b] = _flow(n, lo, length, rng, dev)
        else:
            out[b] = _gaussian(n, lo, length, gamma, rng, dev)
    return out


def _batch_specs(case, seed):
    """Sizes from the case, interactions and traps from the seed."""
    sizes = [s for s in (64, 128, 256, 512) if case["lo"] <= s <= case["hi"]]
    pick = np.random.default_rng(case["count"])
    rng = np.random.default_rng(seed)
    return [dict(n=(s, s), lo=(-12.0, -12.0), length=(24.0, 24.0), g=float(rng.uniform(0, 1000)),
                 gamma=tuple(float(v) for v in rng.uniform(1, 4, size=2)))
            for s in (sizes[int(i)] for i in pick.integers(0, len(sizes), size=case["count"]))]


def _requests(case, seed):
    """A third each 1D, 2D and 3D, a quarter of them in imaginary time."""
    pick = np.random.default_rng(case["count"])
    rng = np.random.default_rng(seed)
    grids = [(4096,), (256, 256), (64, 64, 64), (4096,), (512, 512), (128, 128, 128)]
    out = []
    for i in range(case["count"]):
        n = grids[i % len(grids)]
        imag = i % 4 == 3
        out.append(dict(n=n, lo=(-12.0,) * len(n), length=(24.0,) * len(n), g=float(rng.uniform(0, 500)),
                        gamma=tuple(float(v) for v in rng.uniform(1, 4, size=len(n))), imag=imag,
                        steps=int(pick.integers(case["steps"], 2 * case["steps"] + 1))))
    return out


# ------------------------------------------------------------------ what a program keeps
class _Owned:
    """A handle of the C interface, destroyed with its owner."""

    def __init__(self, handle, destroy):
        self.h, self._destroy = handle, destroy

    def __del__(self):
        self._destroy(self.h)


def prepare(case, seed):
    if case["kind"] == "batch":
        specs = _batch_specs(case, seed)
        rng = np.random.default_rng(seed + 1)
        descs, keep, parts = [], [], []
        for s in specs:
            d, k = gpe.make_desc(s["n"], s["lo"], s["length"], s["g"], DT, s["gamma"])
            descs.append(d)
            keep.append(k)
            parts.append(_gaussian(s["n"], s["lo"], s["length"], s["gamma"], rng, "cuda").to(torch.complex64).reshape(-1))
        flat = torch.cat(parts)
        at = np.concatenate([[0], np.cumsum([p.numel() for p in parts])[:-1]])
        ptrs = [flat.data_ptr() + 8 * int(o) for o in at]
        batch = gpe.gpe_batch_create(descs, torch.cuda.current_stream().cuda_stream)
        return dict(kind="batch", batch=_Owned(batch, gpe.gpe_batch_destroy), flat=flat, ptrs=ptrs, steps=case["steps"])
    if case["kind"] == "serve":
        rng = np.random.default_rng(seed + 1)
        reqs = _requests(case, seed)
        for r in reqs:
            r["desc"], r["keep"] = gpe.make_desc(r["n"], r["lo"], r["length"], r["g"], DT, r["gamma"])
            psi = _gaussian(r["n"], r["lo"], r["length"], r["gamma"], rng, "cuda")
            r["psi"] = psi.to(torch.complex64).cpu().numpy()
            r["out"] = np.empty_like(r["psi"])
        server = gpe.gpe_server_create(16 << 30, 0)
        return dict(kind="serve", server=_Owned(server, gpe.gpe_server_destroy), reqs=reqs)
    lo, length, gamma = _box(case)
    psi = _field(case, seed)
    plan = gpe.Plan(_shape(case), lo, length, g=case["g"], dt=DT, gamma=gamma,
                    prec=gpe.GPE_C64 if case["prec"] == 64 else gpe.GPE_C128, batch=case["batch"])
    if case["kind"] in ("real", "imag"):
        plan.autotune(psi)
    return dict(kind=case["kind"], plan=plan, psi=psi, steps=case.get("steps"), every=case.get("every"))


def run(state):
    kind = state["kind"]
    if kind == "real":
        return state["plan"].step_real(state["psi"], state["steps"])
    if kind == "imag":
        # the single-precision state, the energy too in double
        done, energy = state["plan"].step_imag(state["psi"], state["steps"], 1.0, 0.0, state["every"])
        return [state["psi"], done] if state["psi"].dtype == torch.complex64 else [state["psi"], done, energy]
    if kind == "spectra":
        return state["plan"].spectrum(state["psi"])
    if kind == "energy":
        return [state["plan"].norm_energy(state["psi"]), state["plan"].rms_size(state["psi"])]
    if kind == "batch":
        gpe.gpe_batch_step_real(state["batch"].h, state["ptrs"], state["steps"])
        return state["flat"]
    server = state["server"].h
    tickets = [gpe.gpe_serve_submit(server, r["desc"], r["psi"], imag=r["imag"], nsteps=r["steps"], etol=0.0,
                                    check_every=32) for r in state["reqs"]]
    done = [gpe.gpe_serve_poll(server, t, -1, r["out"]).steps_done for t, r in zip(tickets, state["reqs"])]
    return [[r["out"] for r in state["reqs"]], done]


# ------------------------------------------------------------------ what a pass cannot do without
def _step_flops(n, imag=False):
    """One step: two transforms, the kinetic factor, the nonlinear factor."""
    points = math.prod(n)
    return 2 * 5.0 * points * math.log2(points) + points * (20.0 if imag else 30.0)


def work(case):
    if case["kind"] == "batch":
        specs = _batch_specs(case, 0)
        return dict(bytes=sum(16.0 * math.prod(s["n"]) for s in specs),
                    flops=sum(case["steps"] * _step_flops(s["n"]) for s in specs))
    if case["kind"] == "serve":
        reqs = _requests(case, 0)
        return dict(bytes=sum(16.0 * math.prod(r["n"]) for r in reqs),
                    flops=sum(r["steps"] * _step_flops(r["n"], r["imag"]) for r in reqs))
    n = _shape(case)
    points, size = math.prod(n) * case["batch"], case["prec"] // 8
    if case["kind"] == "spectra":
        return dict(bytes=float(points * size), flops=(1 + 2 * len(n)) * 5.0 * points * math.log2(math.prod(n)))
    if case["kind"] == "energy":
        return dict(bytes=float(points * size), flops=5.0 * points * math.log2(math.prod(n)) + 20.0 * points)
    return dict(bytes=2.0 * points * size, flops=case["batch"] * case["steps"] * _step_flops(n, case["kind"] == "imag"))


# ------------------------------------------------------------------ the same in 64 bits
class _Solver:
    """The scheme in complex128 with torch.fft, in the paper's order."""

    def __init__(self, n, lo, length, gamma, g):
        dev = torch.device("cuda")
        self.n, self.g, self.dim = n, g, tuple(range(len(n)))
        self.dv = math.prod(v / m for v, m in zip(length, n))
        self.x = _coords(n, lo, length, dev)
        self.v = sum(0.5 * (ga * x) ** 2 for ga, x in zip(gamma, self.x))
        d = len(n)
        self.k = [(2 * math.pi * torch.fft.fftfreq(n[a], length[a] / n[a], dtype=torch.float64, device=dev)
                   ).reshape([-1 if i == d - 1 - a else 1 for i in range(d)]) for a in range(d)]
        self.k2 = sum(k * k for k in self.k)

    def half(self, psi, c):
        return psi * torch.exp((self.v + self.g * (psi.real ** 2 + psi.imag ** 2)) * c)

    def kinetic(self, psi, c):
        return torch.fft.ifftn(torch.fft.fftn(psi, dim=self.dim) * torch.exp(self.k2 * c), dim=self.dim)

    def real(self, psi, steps):
        for _ in range(steps):
            psi = self.half(self.kinetic(self.half(psi, -0.5j * DT), -0.5j * DT), -0.5j * DT)
        return psi

    def imag(self, psi, steps):
        for _ in range(steps):
            psi = self.half(self.kinetic(self.half(psi, -0.5 * DT), -0.5 * DT), -0.5 * DT)
            psi = psi / math.sqrt(float((psi.abs() ** 2).sum()) * self.dv)
        return psi

    def energies(self, psi):
        rho = psi.real ** 2 + psi.imag ** 2
        norm = float(rho.sum()) * self.dv
        kin = 0.5 * float((self.k2 * torch.fft.fftn(psi, dim=self.dim).abs() ** 2).sum()) * self.dv / math.prod(self.n)
        pot = float((self.v * rho).sum()) * self.dv
        inter = 0.5 * self.g * float((rho * rho).sum()) * self.dv
        return [norm, kin, pot, inter, kin + pot + inter, (kin + pot + 2 * inter) / norm]

    def sizes(self, psi):
        rho = psi.real ** 2 + psi.imag ** 2
        s2 = [float((x * x * rho).sum() / rho.sum()) for x in self.x]
        return [math.sqrt(s2[a]) if a < len(s2) else 0.0 for a in range(3)] + [math.sqrt(sum(s2))]

    def spectra(self, psi, length, shells):
        d, total = len(self.n), math.prod(self.n)
        hat = torch.fft.fftn(psi, dim=self.dim)
        u, dot = [], 0.0
        for a in range(d):
            k = self.k[a].clone()
            k.reshape(-1)[self.n[a] // 2] = 0.0
            du = torch.fft.ifftn(1j * k * hat, dim=self.dim)
            rho = psi.real ** 2 + psi.imag ** 2
            ua = torch.where(rho >= 1e-30, (psi.conj() * du).imag / rho.sqrt(), torch.zeros_like(rho))
            u.append(torch.fft.fftn(ua + 0j, dim=self.dim))
            dot = dot + self.k[a] * u[-1]
        inv = torch.where(self.k2 > 0, 1 / self.k2, torch.zeros_like(self.k2))
        comp = sum((self.k[a] * dot * inv).abs() ** 2 for a in range(d))
        inc = sum((u[a] - self.k[a] * dot * inv).abs() ** 2 for a in range(d))
        mode = [torch.fft.fftfreq(n, 1.0 / n, dtype=torch.float64, device=hat.device) for n in self.n]
        q2 = sum(((m * (max(length) / v)) ** 2).reshape(k.shape) for m, v, k in zip(mode, length, self.k))
        shell = torch.floor(torch.sqrt(q2) + 0.5).long().expand(hat.shape).reshape(-1)
        out = torch.zeros((2, shells), dtype=torch.float64, device=hat.device)
        for row, e in zip(out, (inc, comp)):
            row.index_add_(0, shell, e.reshape(-1))
        return (0.5 * self.dv / total * out).cpu().numpy()


def exact(case, seed):
    if case["kind"] == "batch":
        rng = np.random.default_rng(seed + 1)
        parts = []
        for s in _batch_specs(case, seed):
            psi = _gaussian(s["n"], s["lo"], s["length"], s["gamma"], rng, "cuda").to(torch.complex64)
            sol = _Solver(s["n"], s["lo"], s["length"], s["gamma"], s["g"])
            parts.append(sol.real(psi.to(torch.complex128), case["steps"]).reshape(-1))
        return torch.cat(parts)
    if case["kind"] == "serve":
        rng = np.random.default_rng(seed + 1)
        out, done = [], []
        for r in _requests(case, seed):
            psi = _gaussian(r["n"], r["lo"], r["length"], r["gamma"], rng, "cuda").to(torch.complex64).to(torch.complex128)
            sol = _Solver(r["n"], r["lo"], r["length"], r["gamma"], r["g"])
            out.append((sol.imag if r["imag"] else sol.real)(psi, r["steps"]).cpu().numpy())
            done.append(None)
        return [out, done]
    n = _shape(case)
    lo, length, gamma = _box(case)
    sol = _Solver(n, lo, length, gamma, case["g"])
    psi = _field(case, seed).to(torch.complex128)
    if case["kind"] == "real":
        return torch.stack([sol.real(p, case["steps"]) for p in psi])
    if case["kind"] == "imag":
        out = torch.stack([sol.imag(p, case["steps"]) for p in psi])
        if case["prec"] == 64:
            return [out, None]
        return [out, None, np.array([sol.energies(p)[4] for p in out])]
    if case["kind"] == "spectra":
        q = math.sqrt(sum((m // 2 * (max(length) / v)) ** 2 for m, v in zip(n, length)))
        shells = int(math.floor(q + 0.5)) + 1
        return np.stack([sol.spectra(p, length, shells) for p in psi], axis=1)
    return [np.array([sol.energies(p) for p in psi]), np.array([sol.sizes(p) for p in psi])]
