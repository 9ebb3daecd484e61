"""What the library's host code launches, without a GPU: its objects linked with a
recording stand-in for the CUDA runtime (fake_cudart.cpp)."""
import ctypes as C
import glob
import importlib.util
import os
import subprocess

import numpy as np
import pytest

from paper_2608_14544_gb300 import build
from paper_2608_14544_gb300 import workloads as wl


class Buf:
    """An address that no launch touches here."""

    def __init__(self, nbytes):
        self.nbytes = int(nbytes)

    def data_ptr(self):
        return 1 << 40

    def numel(self):
        return self.nbytes

    def element_size(self):
        return 1


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    """(bindings over the stand-in, the stand-in's own functions)"""
    build.build()
    objs = [os.path.join(build.BUILD, os.path.basename(s) + ".o") for s in build.sources()]
    if not all(os.path.exists(o) for o in objs):
        build.build(force=True)
    so = str(tmp_path_factory.mktemp("fake") / "libqcl_fake.so")
    cuda = os.path.dirname(os.path.dirname(build._nvcc())) or "/usr/local/cuda"
    here = os.path.dirname(os.path.abspath(__file__))
    subprocess.run(["g++", "-shared", "-fPIC", "-O1", "-std=c++17", "-I",
                    os.path.join(cuda, "include"), os.path.join(here, "fake_cudart.cpp"), *objs,
                    "-o", so, "-Wl,-Bsymbolic", "-lpthread", "-ldl", "-lrt"], check=True)
    spec = importlib.util.spec_from_file_location(
        "paper_2608_14544_gb300.qcl_fake", os.path.join(build.PKG, "qcl.py"))
    q = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(q)
    q.device_buffer = lambda nbytes, device="cuda": Buf(nbytes)
    q._stream_ptr = lambda s=None: None
    lib = q.load(so)
    lib.fake_count.restype = C.c_long
    lib.fake_count.argtypes = lib.fake_max_dyn.argtypes = [C.c_char_p]
    lib.fake_max_dyn.restype = C.c_ulong
    return q, lib


def _lvc(ns, n):
    rng = np.random.default_rng(2)
    a = rng.uniform(0, 0.1, (n, ns, ns))
    return wl._model(np.diag(0.4 * np.arange(ns)), a + a.transpose(0, 2, 1), np.ones(n),
                     rng.uniform(0.5, 2.0, n))


@pytest.mark.parametrize("ns,n,kernel,dyn", [
    (2, 100, b"k_bulk2_split2", 102_400), (3, 60, b"k_bulkN", 64 * 480), (4, 32, b"k_bulkN", 32_768),
    (4, 64, b"k_bulkN", 32_768), (5, 200, b"k_bulkN", 14_000), (8, 256, b"k_bulkN", 40_000)])
def test_solves_on_a_second_device(fake, ns, n, kernel, dyn):
    """A kernel's shared-memory limit is raised on every device it runs on."""
    q, lib = fake
    model = (wl.spin_boson(0.5, 0.5, *wl.ohmic_modes(n, 0.3, 2.5)) if ns == 2 else _lvc(ns, n))
    try:
        for device in (0, 1, 0):
            lib.cudaSetDevice(device)
            lib.fake_reset()
            r = q.Run(q.Model(model), 100_000, 1, q.PREC_FP32_BULK, 3)
            r.propagate(4, 0.01, 2)
            assert lib.fake_count(kernel) >= 1
            assert lib.fake_max_dyn(kernel) >= dyn
    finally:
        lib.cudaSetDevice(0)


@pytest.mark.parametrize("ns,n", [(3, 40), (8, 256)])
def test_spawning_on_a_second_device(fake, ns, n):
    q, lib = fake
    try:
        for device in (0, 1):
            lib.cudaSetDevice(device)
            lib.fake_reset()
            r = q.SpawnRun(q.Model(_lvc(ns, n)), 100, 1000, 1, 3, precision=q.PREC_FP32_BULK)
            r.propagate(4, 0.01, 2)
            assert lib.fake_max_dyn(b"k_spawnN_step32") > 0
    finally:
        lib.cudaSetDevice(0)


def test_a_refused_limit_is_the_calls_error(fake):
    """No kernel runs in place of the refused one, and none on what it would have
    written."""
    q, lib = fake
    lib.fake_refuse_limits(1)
    try:
        lib.fake_reset()
        spawn = q.SpawnRun(q.Model(_lvc(8, 256)), 100, 1000, 1, 3, precision=q.PREC_FP32_BULK)
        with pytest.raises(q.QclError, match="launch failed"):
            spawn.propagate(1, 0.01, 2)
        assert lib.fake_count(b"k_spawn_scan") == lib.fake_count(b"k_spawnN_scatter32") == 0
        for model in (_lvc(4, 64), wl.spin_boson(0.5, 0.5, *wl.ohmic_modes(100, 0.3, 2.5))):
            run = q.Run(q.Model(model), 300_000, 1, q.PREC_FP32_BULK, 3)
            with pytest.raises(q.QclError, match="launch failed"):
                run.propagate(4, 0.01, 2)
        assert lib.fake_count(b"k_bulk") == 0
    finally:
        lib.fake_refuse_limits(0)


@pytest.mark.parametrize("ns,n,rep,walkers,steps,least,most", [
    (2, 1, "adiabatic", 10_000, 600, 3, 3), (2, 3, "adiabatic", 1_000_000, 512, 2, 2),
    (2, 256, "adiabatic", 10_000_000, 256, 100, 256), (2, 100, "diabatic", 3_000_000, 256, 5, 64),
    (4, 6, "adiabatic", 20_000, 32, 2, 2), (4, 6, "diabatic", 1_000_000, 32, 2, 2),
    (8, 256, "adiabatic", 1_000_000, 32, 32, 32), (4, 40, "adiabatic", 1_000_000, 32, 8, 32)])
def test_fp64_launches_follow_the_work_of_a_step(fake, ns, n, rep, walkers, steps, least, most):
    """Small solves take many steps a launch; one of 1e7 walkers and 256 modes,
    whose step takes a tenth of a second, takes few."""
    q, lib = fake
    model = wl.random_lvc2(n, 3, 0.3) if ns == 2 else _lvc(ns, n)
    r = q.Run(q.Model(dict(model, repr=rep)), walkers, 1, q.PREC_FP64, 2)
    lib.fake_reset()
    r.propagate(steps, 0.01, 1000)
    kernel = b"k_steps_f64" if ns == 2 else (b"k_stepsN_dia_f64" if rep == "diabatic"
                                            else b"k_stepsN_f64")
    assert least <= lib.fake_count(kernel) <= most
