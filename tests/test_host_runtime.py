"""Host code of the library on a CUDA runtime without a GPU (fake_cudart.cpp): the
paths of a call that its kernels' results do not depend on."""

import ctypes
import glob
import os
import re
import shutil
import subprocess

import numpy as np
import pytest

from paper_2501_12928_gb300 import _build, beor

HERE = os.path.dirname(os.path.abspath(__file__))
HEADER = os.path.join(os.path.dirname(HERE), "include", "beor.h")
STREAM = 0x1000   # any stream but the null one


@pytest.fixture(scope="module")
def fake_library(tmp_path_factory):
    if shutil.which("g++") is None or (shutil.which("nvcc") is None and not os.path.exists(_build._nvcc())):
        pytest.skip("no compiler")
    objs = [os.path.join(_build.OUT_DIR, s.replace(".cu", ".o")) for s in _build.SOURCES]
    newest = max(map(os.path.getmtime, glob.glob(os.path.join(_build.CSRC, "*")) + [_build.__file__, HEADER]))
    if not all(os.path.exists(o) and os.path.getmtime(o) > newest for o in objs):
        _build.build()
    lib = str(tmp_path_factory.mktemp("fake") / "libbeor_fake.so")
    include = os.path.join(os.path.dirname(os.path.dirname(_build._nvcc())) or "/usr/local/cuda", "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-Wl,-Bsymbolic", "-I", include, "-o", lib,
                    os.path.join(HERE, "fake_cudart.cpp"), *objs], check=True)
    return lib


@pytest.fixture
def fake(fake_library, tmp_path, monkeypatch):
    """The package on a copy of its own, so that nothing is left from another test."""
    monkeypatch.setattr(beor, "LIB_PATH", shutil.copy(fake_library, tmp_path))
    lib = beor._load()
    lib.fake_log.restype = ctypes.c_char_p
    lib.fake_used.restype = ctypes.c_size_t
    lib.fake_set_total.argtypes = [ctypes.c_int, ctypes.c_size_t]
    monkeypatch.setattr(beor, "lib", lib)
    return lib


class Array:
    """Device memory with what the package asks of a tensor."""

    def __init__(self, lib, device, nbytes, offset=0):
        p = ctypes.c_void_p()
        lib.cudaSetDevice(device)
        assert lib.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(nbytes)) == 0
        self.address = p.value + offset


def _copies(lib, key, address):
    """Copies from (key 2) or to (key 1) an address: their sizes."""
    rows = [r.split() for r in lib.fake_log().decode().splitlines() if r.startswith("copy")]
    return [int(r[3]) for r in rows if int(r[key]) == address]


N_IN, N = 3, 5000


@pytest.mark.parametrize("where_x, where_y, copies", [
    ("own", "own", (0, 0)), ("other", "own", (1, 0)), ("own", "other", (0, 1)), ("host", "own", (1, 0)),
    ("own", "head of x", (0, 1)), ("own", "last of x", (0, 1)), ("own", "behind x", (0, 0)), ("odd", "odd", (1, 1))])
def test_predictions_in_place_only_where_the_kernel_may(fake, where_x, where_y, copies):
    """The kernel addresses the caller's arrays only if they are its own device's,
    aligned and apart; otherwise inputs and predictions are copied."""
    em = beor.Emulator(N_IN, 16, 1, device=0)
    x_bytes, host = 4 * N_IN * N, np.zeros((N, N_IN), np.float32)
    base = Array(fake, 1 if where_x == "other" else 0, x_bytes + 4 * N + 4, 1 if where_x == "odd" else 0)
    x = host.ctypes.data if where_x == "host" else base.address
    y = {"head of x": x, "last of x": x + x_bytes - 4, "behind x": x + x_bytes}.get(where_y) or Array(
        fake, 1 if where_y == "other" else 0, 4 * N + 4, 1 if where_y == "odd" else 0).address
    fake.fake_clear_log()
    assert fake.beor_mlp_infer(em._h, x, N, y, STREAM) == 0
    assert _copies(fake, 2, x) == [x_bytes] * copies[0]
    assert _copies(fake, 1, y) == [4 * N] * copies[1]
    assert re.search("launch 0 .*rows_kernel", fake.fake_log().decode())


def _like(lib, n=140, n_vis=200, precision="mixed", device=0):
    from synth.instrument import random_problem
    p = random_problem(n_vis, n, 3, seed=n)
    lk = beor.Likelihood(precision, device)
    lk.set_T(p["T"], p["kbin"], 3, 2.0)
    lk.set_data(p["d"], p["noise_var"])
    lk.precompute(STREAM)
    return lk, p


@pytest.mark.parametrize("where, copied", [("own", False), ("own, 8 bytes on", True), ("other", True), ("host", True)])
def test_normal_matrix_stored_by_the_kernel_only_where_it_may(fake, where, copied):
    """16-byte stores go to 16-byte aligned memory of the context's own device; a
    beor_c128 is aligned to 8 bytes, and other memory takes a copy."""
    lk, p = _like(fake)
    n = p["T"].shape[1]
    host = np.zeros((n, n), np.complex128)
    out = host.ctypes.data if where == "host" else Array(fake, where == "other", 16 * n * n + 8, 8 * ("8" in where)).address
    fake.fake_clear_log()
    assert fake.beor_get_M(lk._h, out) == 0
    assert _copies(fake, 1, out) == [16 * n * n] * copied
    assert "unpack_hermitian" in fake.fake_log().decode()


def _kernels(lib, device):
    return re.findall(rf"launch {device} (\S+)", lib.fake_log().decode())


@pytest.mark.parametrize("first", [0, 1])
def test_emulators_on_two_devices(fake, first):
    """A second device allows the kernels their shared memory too, and the split of
    the rows follows its own number of SMs."""
    rows = np.zeros((4000, N_IN), np.float32)
    for device in (first, 1 - first):
        fake.fake_clear_log()
        for depth in (1, 8):
            em = beor.Emulator(N_IN, 32, depth, device=device)
            for n in (16, 4000):
                em.train_step(rows[:n], np.zeros(n, np.float32), 1e-3, stream=STREAM)
                em.infer(rows[:n], stream=STREAM)
        wide = "rows_kernelILi4ELi2ELb0E"   # 64 rows a CTA: beyond 16 rows on each half of 76 SMs, not of 152
        assert any(wide in k for k in _kernels(fake, device)) == (device == 1)
        assert not _kernels(fake, 1 - device)


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
@pytest.mark.parametrize("first", [0, 1])
def test_likelihoods_on_two_devices(fake, first, precision):
    """The same for the likelihood's kernels, in batches of each size class."""
    for device in (first, 1 - first):
        lk, p = _like(fake, 300, 400, precision, device)
        for B in (1, 20, 70, 200):
            phi = np.zeros((B, 3))
            lk.lnl(phi, stream=STREAM)
            lk.lnl(phi, stream=STREAM)
        lk.posterior_mean(np.zeros(3), stream=STREAM)
        assert _kernels(fake, device)


def _idle_batch(lib):
    """A context with new data and the idle batch of an earlier evaluation; its bytes."""
    lk, p = _like(lib)
    before = lib.fake_used(0)
    lk.lnl(np.zeros((8, 3)), stream=STREAM)
    batch = lib.fake_used(0) - before
    lk.set_data(p["d"], p["noise_var"])
    return lk, p, batch


def _set_instrument(lk, p):
    geometry = dict(nu=7, nf=12, nf_grid=0, n_pix=64, n_k=3, f0_hz=1.5e8, df_hz=1e6, beam_fwhm_rad=0.2, latitude_rad=-0.5,
                    lssm_prior_var=2.0, bl_enu_m=np.random.default_rng(0).uniform(-30, 30, (200, 3)),
                    hour_angle_rad=np.linspace(-0.1, 0.1, 4))
    beor.Likelihood("fp64").set_instrument_desc(geometry)


@pytest.mark.parametrize("call", [
    lambda lk, p: lk.precompute(STREAM),                       # digit planes of the dense precompute
    lambda lk, p: beor.Emulator(9, 256, 8),
    _set_instrument,
    lambda lk, p: beor.Likelihood("mixed").set_T(np.ones((1000, 300)), np.zeros(300, np.int32), 1, 2.0)])
def test_allocations_get_the_idle_batches_memory(fake, call):
    """On a full device, whatever the library allocates."""
    lk, p, batch = _idle_batch(fake)
    used = fake.fake_used(0)
    fake.fake_set_total(0, used + (1 << 20))
    call(lk, p)
    assert fake.fake_used(0) < used + (1 << 20) and batch > 4 << 20


def test_idle_batches_leave_memory_to_others(fake):
    """They are kept on a device with room, and not beyond a sixteenth of it or
    beyond what is free beside them."""
    lk, p, batch = _idle_batch(fake)

    def kept(free, total=None):
        lk.precompute(STREAM)
        lk.lnl(np.zeros((8, 3)), stream=STREAM)
        used = fake.fake_used(0)
        ballast = Array(fake, 0, total - free - used) if total else None
        fake.fake_set_total(0, total or used + free)
        before = fake.fake_used(0)
        lk.set_data(p["d"], p["noise_var"])
        idle = before - fake.fake_used(0) < batch // 2
        fake.fake_set_total(0, 1 << 38)
        if ballast:
            fake.cudaFree(ctypes.c_void_p(ballast.address))
        return idle

    assert kept(20 * batch)
    assert not kept(4 * batch)                       # more than a sixteenth
    assert kept(2 * batch, total=64 * batch)
    assert not kept(batch // 2, total=64 * batch)    # more than what is free


def test_rejected_points_leave_an_idle_batch_idle(fake):
    """Points that are refused are no evaluation of the new data: the wait for one
    still reports that there is none, and the batch's memory is still given back."""
    lk, p, batch = _idle_batch(fake)
    lk.precompute(STREAM)
    for B in (8, 5):   # an idle batch, and a shape that has none
        phi = np.zeros((B, 3))
        phi[-1, 1] = np.nan
        with pytest.raises(beor.BeorError, match="invalid argument"):
            lk.lnl(phi, stream=STREAM)
        with pytest.raises(beor.BeorError, match="out of order"):
            beor.lnl_multi_wait([lk], [B], 0, STREAM)
    used = fake.fake_used(0)
    fake.fake_set_total(0, used)
    beor.Emulator(9, 256, 8)
    assert fake.fake_used(0) < used
    fake.fake_set_total(0, 1 << 38)
    lk.lnl(np.zeros((8, 3)), stream=STREAM)
    beor.lnl_multi_wait([lk], [8], 0, STREAM)


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_work_waits_for_the_null_streams(fake, precision):
    """Buffers that the library fills on the null stream are filled before it works
    with them on the caller's, which need not wait for the null stream: first calls of
    a shape, batches taken up again, growing emulator batches."""
    lk, p = _like(fake, 140, 200, precision)
    lk.lnl(np.zeros((8, 3)), stream=STREAM)
    lk.posterior_mean(np.zeros(3), stream=STREAM)
    lk.set_data(p["d"], p["noise_var"])
    lk.precompute(STREAM)
    lk.lnl(np.zeros((8, 3)), stream=STREAM)
    em = beor.Emulator(N_IN, 32, 2)
    for n in (100, 3000, 9000):
        em.infer(np.zeros((n, N_IN), np.float32), stream=STREAM)
        em.train_step(np.zeros((n, N_IN), np.float32), np.zeros(n, np.float32), 1e-3, stream=STREAM)
    assert fake.fake_unordered() == 0


def test_no_evaluation_after_a_failed_precompute(fake):
    """A precompute that runs out of memory leaves matrices of which some are the new
    data's: there is nothing to evaluate until one succeeds."""
    lk, p = _like(fake)
    fake.fake_set_total(0, fake.fake_used(0) + (1 << 20))
    with pytest.raises(beor.BeorError, match="out of memory"):
        lk.precompute(STREAM)
    fake.fake_set_total(0, 1 << 38)
    for call in (lambda: lk.lnl(np.zeros((1, 3)), stream=STREAM), lambda: lk.posterior_mean(np.zeros(3), stream=STREAM),
                 lk.get_M, lk.get_dbar):
        with pytest.raises(beor.BeorError, match="out of order"):
            call()
    lk.precompute(STREAM)
    lk.lnl(np.zeros((1, 3)), stream=STREAM)


@pytest.mark.parametrize("short", [1, 300, 1000, 3000, 100000, 1 << 22])
def test_a_batch_that_does_not_fit_is_out_of_memory(fake, short):
    """Whichever of its allocations fails, the tile lists' at the end among them; the
    shape works once there is room."""
    lk, p = _like(fake)
    before = fake.fake_used(0)
    lk.lnl(np.zeros((8, 3)), stream=STREAM)
    batch = fake.fake_used(0) - before
    lk, p = _like(fake)
    fake.fake_set_total(0, fake.fake_used(0) + batch - short)
    with pytest.raises(beor.BeorError, match="out of memory"):
        lk.lnl(np.zeros((8, 3)), stream=STREAM)
    fake.fake_set_total(0, 1 << 38)
    lk.lnl(np.zeros((8, 3)), stream=STREAM)
