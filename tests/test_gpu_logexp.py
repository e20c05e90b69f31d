"""logexp.cuh's logarithm, exponential, square root and quotient against 200-bit arithmetic, with
CUDA's functions where they hand over, and the FP64 saturation temperature against the six-step
Newton iteration."""
import ctypes
import os
import shutil
import subprocess
import tempfile

import numpy as np
import pytest

torch = pytest.importorskip("torch")
mp = pytest.importorskip("mpmath")

from conftest import ROOT

pytestmark = pytest.mark.gpu
SPECIAL = np.array([0.0, -0.0, -1.0, np.inf, -np.inf, np.nan, 5e-324, 1e-310, 2.2250738585072014e-308, 1.7976931348623157e308,
                    -1e-300, 1e300, 2.0 ** -1000, 2.0 ** 1000, 700.0, -700.0, 709.0, -745.0, 1000.0, -1000.0])


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    so = os.path.join(tempfile.mkdtemp(), "logexp_check.so")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "--expt-relaxed-constexpr", "-shared",
                    "-Xcompiler", "-fPIC", "-o", so, os.path.join(ROOT, "tests", "kernels", "logexp_check.cu")], check=True)
    L = ctypes.CDLL(so)
    L.logexp_check.argtypes = [ctypes.c_int] + [ctypes.c_void_p] * 4 + [ctypes.c_int]

    def run(which, x, y=None):
        X = torch.tensor(np.asarray(x, dtype=np.float64), device="cuda")
        Y = X if y is None else torch.tensor(np.asarray(y, dtype=np.float64), device="cuda")
        R, D = torch.empty_like(X), torch.empty_like(X)
        torch.cuda.synchronize()
        assert L.logexp_check(which, X.data_ptr(), Y.data_ptr(), R.data_ptr(), D.data_ptr(), X.numel()) == 0
        return R.cpu().numpy(), D.cpu().numpy()

    return run


def _error(got, exact):
    with mp.workprec(200):
        return np.array([float(abs(mp.mpf(float(g)) - e)) for g, e in zip(got, exact)])


def _exact(f, x):
    with mp.workprec(200):
        return [f(mp.mpf(float(v))) for v in x]


def _ulp(exact):
    return np.array([np.spacing(abs(float(e))) for e in exact])


# Bounds: the last addition's half ulp, plus the FP32 tail (log: r^3/3 <= 3.2e-10 of FP32 relative
# error 3 x 2^-23, 1.2e-16, and the low parts; exp, expm1: far below an ulp) and the roundings of
# the leading terms: 1 ulp + 1.2e-16 for log, 1.5 ulp for exp, 2 ulp for expm1.
def test_log(lib):
    g = np.random.default_rng(1)
    x = np.concatenate([150 + 400 * g.random(4000), np.exp(-70 + 90 * g.random(4000)), 1 + 0.1 * (g.random(4000) - 0.5),
                        2.0 ** np.arange(-1022, 1023, 7), np.nextafter(2.0 ** np.arange(-20.0, 20.0), 0),
                        1024.0 / (512 + np.arange(512) + 0.5)])
    got, _ = lib(0, x)
    e = _exact(mp.log, x)
    assert np.all(_error(got, e) <= _ulp(e) + 1.2e-16)
    got, ref = lib(0, SPECIAL)
    assert np.array_equal(got[:9], ref[:9], equal_nan=True)


@pytest.mark.parametrize("which,f,bound", [(1, mp.exp, 1.5), (2, mp.expm1, 2.0)])
def test_exp(lib, which, f, bound):
    g = np.random.default_rng(2)
    x = np.concatenate([-699 + 1398 * g.random(4000), -30 + 60 * g.random(4000), 0.02 * (g.random(4000) - 0.5),
                        np.log(2) / 512 * (np.arange(-600, 600) + 0.5), 10.0 ** np.arange(-300, 0), -(10.0 ** np.arange(-300, 0))])
    got, _ = lib(which, x)
    e = _exact(f, x)
    assert np.all(_error(got, e) <= bound * _ulp(e))
    got, ref = lib(which, SPECIAL)
    hand = ~(np.abs(SPECIAL) < 700)
    assert np.array_equal(got[hand], ref[hand], equal_nan=True)


def test_sqrt_and_quotient(lib):
    g = np.random.default_rng(3)
    x, y = np.exp(-300 + 600 * g.random(8000)), np.exp(-300 + 600 * g.random(8000)) * np.where(g.random(8000) < 0.5, -1, 1)
    got, ref = lib(3, x)
    assert np.all(np.abs(got - ref) <= 2 * np.spacing(ref))
    got, ref = lib(4, x, y)
    ok = np.isfinite(ref) & (np.abs(ref) > 1e-290)
    assert np.all(np.abs(got - ref)[ok] <= 3 * np.spacing(np.abs(ref[ok])))
    got, ref = lib(3, SPECIAL)
    same = ~((SPECIAL >= 2.0 ** -1000) & (SPECIAL < 2.0 ** 1000))
    assert np.array_equal(got[same], ref[same], equal_nan=True)
    b = SPECIAL
    got, ref = lib(4, np.full(b.size, 3.0), b)
    same = ~((np.abs(b) >= 2.0 ** -1000) & (np.abs(b) < 2.0 ** 1000))
    assert np.array_equal(got[same], ref[same], equal_nan=True)


def test_conversion_and_halving_are_exact(lib):
    g = np.random.default_rng(4)
    x = np.concatenate([g.integers(0, 1 << 32, 4096, dtype=np.uint32).view(np.float32).astype(np.float64), [0.0, -0.0, np.inf, 1e-45, 1.0]])
    got, ref = lib(5, x)
    assert np.array_equal(got, ref, equal_nan=True)
    x = np.concatenate([np.exp(-600 + 1200 * g.random(4096)), [0.0, -3.0, np.inf, -np.inf, np.nan]])
    got, ref = lib(6, x)
    assert np.array_equal(got, ref, equal_nan=True)


# The root's condition: rounding of ln p (a few ulp of its largest term, 30 to 100: 1e-14) over the
# curve's slope, 0.03 to 1.7 per K: 3e-13 K.
@pytest.mark.parametrize("which", [7, 8])
def test_saturation_temperature(lib, which):
    lnpv = np.concatenate([np.linspace(-69.0, 12.0, 5000), np.log(np.linspace(0.1, 4000.0, 5000))])
    got, ref = lib(which, lnpv)
    assert np.all(np.isfinite(got)) and np.abs(got - ref).max() <= 5e-13
