"""What the library's host code asks of the CUDA runtime, and in which order, against
a stand-in for the runtime (fake_cudart.cpp; no GPU, no kernel runs)."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
STREAM = 0x1000                      # a stream of the caller's: only its number counts
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")


class Fake:
    def __init__(self, lib):
        self.lib = lib
        lib.fake_log.restype = ctypes.c_char_p
        lib.fake_live_bytes.restype = ctypes.c_size_t

    def log(self):
        return self.lib.fake_log().decode().splitlines()


@pytest.fixture(scope="module")
def loaded(tmp_path_factory):
    import paper_2301_08275_gb300 as gpe
    from paper_2301_08275_gb300 import buildlib
    gpe.build()
    path = str(tmp_path_factory.mktemp("fake") / "libgpe_fake.so")
    objs = [os.path.join(buildlib.BUILD, s.replace(".cu", ".o")) for s in buildlib.SOURCES]
    # (symbolic: another runtime that is loaded already must not take the calls)
    subprocess.run(["g++", "-O1", "-std=c++17", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-I" + os.path.join(CUDA, "include"),
                    os.path.join(HERE, "fake_cudart.cpp")] + objs + ["-o", path, "-lpthread"], check=True)
    real = gpe.LIB_PATH, gpe._lib
    gpe.LIB_PATH, gpe._lib = path, None
    try:
        yield gpe, Fake(gpe.lib())
    finally:
        gpe.LIB_PATH, gpe._lib = real
        os.unlink(path)


@pytest.fixture
def unused(loaded, tmp_path):
    """Another copy of the library, none of whose kernels has been asked for yet."""
    gpe = loaded[0]
    path = str(tmp_path / "libgpe_unused.so")
    shutil.copy(gpe.LIB_PATH, path)
    before = gpe.LIB_PATH, gpe._lib
    gpe.LIB_PATH, gpe._lib = path, None
    try:
        yield gpe, Fake(gpe.lib())
    finally:
        gpe.LIB_PATH, gpe._lib = before
        os.unlink(path)


@pytest.fixture
def gpe(loaded):
    return loaded[0]


@pytest.fixture
def fake(loaded):
    loaded[1].lib.fake_reset()
    return loaded[1]


def desc(gpe, n, prec=0, gamma=1.0, batch=1, V=None):
    d = len(n)
    return gpe.make_desc(n, (-6.0,) * d, (12.0,) * d, g=10.0, dt=1e-3, gamma=None if V is not None else (gamma,) * d,
                         prec=prec, batch=batch, V=V)


class Made:
    """A plan on STREAM and a state for it."""

    def __init__(self, gpe, n, prec=0, gamma=1.0, batch=1, V=None):
        self.gpe = gpe
        self.d, self.keep = desc(gpe, n, prec, gamma, batch, V)
        self.batch = batch
        self.h = gpe.gpe_plan_create(self.d, STREAM)
        # (16 bytes aligned)
        self.buf = np.zeros(2 * int(np.prod(n)) * batch + 2, dtype=np.float64)
        self.psi = (self.buf.ctypes.data + 15) // 16 * 16

    def __enter__(self):
        return self

    def __exit__(self, *exc):
        self.gpe.gpe_plan_destroy(self.h)


def unordered(log):
    """Lines of work on a stream of its own while work of the default stream (whose
    calls may return before it is done, and which such a stream does not wait for)
    has not been waited for."""
    pending, out = False, []
    for line in log:
        what, _, rest = line.partition(" ")
        s = rest.split(" ")[0]
        if line in ("wait 0", "wait all"):
            pending = False
        elif what in ("copy", "set") and s == "0":
            pending = True
        elif what in ("copy", "set", "kernel") and pending:
            out.append(line)
    return out


@pytest.mark.parametrize("prec", [0, 1], ids=["c64", "c128"])
@pytest.mark.parametrize("n", [(4096,), (64, 64), (128, 256), (128, 128, 64)], ids=lambda n: "x".join(map(str, n)))
def test_uploads_are_complete_before_the_plan_stream_runs(gpe, fake, n, prec):
    with Made(gpe, n, prec) as p:
        gpe.gpe_step_real(p.h, p.psi, 2)
        gpe.gpe_step_imag(p.h, p.psi, 2, 1.0, 0.0, 1, 1)
        gpe.gpe_norm_energy(p.h, p.psi, 1)
        gpe.gpe_spectrum(p.h, p.psi, 15, 1)
    assert any(line.startswith("kernel") for line in fake.log())
    assert unordered(fake.log()) == []


@pytest.mark.parametrize("graph", [0, 1])
def test_batch_uploads_are_complete_before_the_groups_run(gpe, fake, graph):
    ns = [(64, 64), (64, 64), (256, 128), (128, 128, 64)]
    made = [desc(gpe, n) for n in ns]
    bufs = [np.zeros(2 * int(np.prod(n)) + 2) for n in ns]
    ptrs = [(b.ctypes.data + 15) // 16 * 16 for b in bufs]
    b = gpe.gpe_batch_create([m[0] for m in made], STREAM)
    gpe.gpe_batch_step_real(b, ptrs, 2, graph)
    gpe.gpe_batch_step_real(b, ptrs[1::-1] + ptrs[2:], 2, graph)
    gpe.gpe_batch_norm_energy(b, ptrs)
    gpe.gpe_batch_destroy(b)
    assert unordered(fake.log()) == []


SPEC_PLANS = [((64, 128), 0), ((64, 128), 1), ((32, 64), 0), ((64, 64, 128), 0), ((512,), 1)]


@pytest.mark.parametrize("n,prec", SPEC_PLANS, ids=lambda v: str(v))
def test_spectra_after_a_failed_allocation(gpe, fake, n, prec):
    """Whichever of a first spectrum's allocations fails, a later call makes the rest:
    as many bytes live on the device as after a first call that met no failure."""
    sizes = []
    for k in range(12):
        with Made(gpe, n, prec) as p:
            start = fake.lib.fake_live_bytes()
            fake.lib.fake_fail_alloc(k)
            if k:
                try:
                    gpe.gpe_spectrum(p.h, p.psi, 15, 1)
                except gpe.GpeError as e:
                    assert e.status in (3, 4)
                else:
                    break
            fake.lib.fake_fail_alloc(0)
            gpe.gpe_spectrum(p.h, p.psi, 15, 1)
            sizes.append(fake.lib.fake_live_bytes() - start)
    assert len(sizes) > 4 and len(set(sizes)) == 1


def test_spectra_of_two_threads_ask_for_one_shared_memory_size(gpe, fake):
    """The size a kernel may take is the process's, not the call's: a call that set
    a smaller one could take it from another thread's launch."""
    for n in ((64, 64), (128, 64)):
        with Made(gpe, n) as p:
            for kinds in (3, 4):
                gpe.gpe_spectrum(p.h, p.psi, kinds, 1)
    got = {line for line in fake.log() if line.startswith("resolve") and "k_bin" in line}
    assert len(got) == 1


def timed(gpe, fake, p):
    """Sweeps that gpe_plan_autotune launches."""
    fake.lib.fake_reset()
    gpe.gpe_plan_autotune(p.h, p.psi, 1, 0)
    return sum(line.startswith("kernel") and "k_pass" in line for line in fake.log())


def test_tuner_remembers_by_the_kind_of_potential(gpe, fake):
    """Row sweeps with a trap, without one and with a sampled potential are different
    kernels: a choice made for one is not the others'."""
    n = (512, 32)
    V = np.zeros((32, 512))
    kinds = [dict(gamma=1.0), dict(gamma=0.0), dict(V=V)]
    for kw in kinds:
        with Made(gpe, n, **kw) as p:
            assert timed(gpe, fake, p) > 0
    for kw in kinds:
        with Made(gpe, n, **kw) as p:
            assert timed(gpe, fake, p) == 0
            gpe.gpe_plan_set_option(p.h, gpe.GPE_OPT_GENERIC_PASSES, 1)
            assert timed(gpe, fake, p) > 0


@pytest.mark.parametrize("clusters", [8, 0])
def test_tuner_times_the_sweeps_of_planes_stepped_on_chip(gpe, fake, clusters):
    """Trap schedules and diagnostics of such a plan are sweeps, and so are all its
    steps where no cluster of that size can be placed."""
    fake.lib.fake_clusters(clusters)
    with Made(gpe, (128, 64 if clusters else 128)) as p:
        assert timed(gpe, fake, p) > 0


BATCHES = {"resident": [((64, 64), 0)], "plane": [((64, 64), 1)], "sweeps": [((128, 128), 1)] * 9, "rows": [((512, 16), 0)],
           "3d": [((128, 64, 16), 0)], "3d_c128": [((64, 128, 16), 1)], "lines": [((1024,), 0)], "few_lines": [((128,), 1)],
           "many_lines": [((32,), 1)] * 310}


@pytest.mark.parametrize("kind", BATCHES)
def test_batch_resolves_its_kernels_before_capture(unused, kind):
    gpe, fake = unused
    made = [desc(gpe, n, prec) for n, prec in BATCHES[kind]]
    bufs = [np.zeros(2 * int(np.prod(n)) + 2) for n, _ in BATCHES[kind]]
    b = gpe.gpe_batch_create([m[0] for m in made], STREAM)
    fake.lib.fake_reset()
    gpe.gpe_batch_step_real(b, [(x.ctypes.data + 15) // 16 * 16 for x in bufs], 3, 1)
    gpe.gpe_batch_destroy(b)
    log = fake.log()
    captured = log[log.index("begin"):log.index("end")]
    assert any(line.startswith("kernel") for line in captured)
    assert not [line for line in captured if line.startswith("resolve")]


@pytest.mark.parametrize("prec", [0, 1], ids=["c64", "c128"])
@pytest.mark.parametrize("n", [(64,), (32, 64), (32, 16, 8)], ids=lambda n: "x".join(map(str, n)))
def test_admission_waits_for_the_stream_once(gpe, fake, n, prec):
    """Parameters and tables of a slot are uploaded without a wait between them."""
    d, keep = desc(gpe, n, prec)
    psi = np.zeros(n[::-1], dtype=np.complex128 if prec else np.complex64)
    srv = gpe.gpe_server_create(1 << 30, max_active=4, chunk_steps=4)
    t = gpe.gpe_serve_submit(srv, d, psi, imag=False, nsteps=3)
    assert gpe.gpe_serve_poll(srv, t, -1, np.empty_like(psi)).status == 0
    gpe.gpe_server_destroy(srv)
    log = fake.log()
    first = next(i for i, line in enumerate(log) if line.startswith("kernel"))
    stream = log[first].split()[1]
    assert log[:first].count("wait " + stream) == 1
