"""Kernels with more than 48 KB of dynamic shared memory are opted in on every device that launches
them: the library's own objects, linked against a stand-in for the CUDA runtime with two devices."""
import ctypes as C
import os
import subprocess

import pytest

from conftest import ROOT


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    from paper_2504_20742_gb300 import _lib, build
    build.build()
    objs = [os.path.join(build.BUILD, s.replace(".cu", ".o")) for s in build.SOURCES]
    so = str(tmp_path_factory.mktemp("fake") / "libfake.so")
    include = os.path.join(os.path.dirname(os.path.dirname(build._nvcc())), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-Wl,-Bsymbolic", "-I" + include, "-o", so,
                    os.path.join(ROOT, "tests", "kernels", "fake_cudart.cpp"), *objs], check=True)
    L = C.CDLL(so)
    for name, (res, args) in _lib._SIGS.items():
        getattr(L, name).restype, getattr(L, name).argtypes = res, args
    return L


def _both_devices(L, call):
    """call() on device 0 twice, then on device 1: every launch is within its device's limit."""
    for dev in (0, 0, 1):
        L.fake_device(dev)
        n, r = L.fake_launches(), L.fake_refused()
        status = call()
        assert status == 0, (dev, L.ct_last_error())
        assert L.fake_launches() > n and L.fake_refused() == r
    L.fake_device(0)


@pytest.fixture()
def buf():
    b = (C.c_char * (1 << 22))()
    p = C.addressof(b)
    yield p + (-p % 256)


def test_inference(fake, buf):
    _both_devices(fake, lambda: fake.ct_mlp_infer(buf, buf, 1000, buf, buf, None))


def test_training_kernels(fake, buf):
    n = 3000
    wb = fake.ct_mlp_work_bytes(n)
    _both_devices(fake, lambda: fake.ct_mlp_loss_grad(buf, buf, buf, buf, n, buf, buf, buf, wb, None))
    _both_devices(fake, lambda: fake.ct_mlp_loss_grad_tc(buf, buf, buf, buf, n, buf, buf, buf, buf, wb, None))


@pytest.mark.parametrize("prec", [0, 1])
def test_steps(fake, buf, prec):
    from paper_2504_20742_gb300 import _lib
    from synth import cases
    c = _lib._case(cases.plume_case(nx=256, nr=128)[0])
    _both_devices(fake, lambda: fake.ct_step(C.byref(c), prec, buf, buf + 64, buf, 1, 0.5, None))


def test_surrogate_steps(fake, buf):
    from paper_2504_20742_gb300 import _lib
    from synth import cases
    c = _lib._case(cases.plume_case(nx=256, nr=128)[0])
    for shape in (0, 9):                                  # the fused tile, the column sweep and its queue
        assert fake.ct_set_tile_shape(C.byref(c), 2, shape) == 0
        _both_devices(fake, lambda: fake.ct_step_surrogate(C.byref(c), buf, buf + 64, buf, buf, 1, 0.5, None))
    fake.ct_set_tile_shape(C.byref(c), 2, -1)
