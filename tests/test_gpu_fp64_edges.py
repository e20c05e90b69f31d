"""FP64 source arithmetic where its fast forms reach the end of their range: the saturation
temperature of the tabulated curves beyond the tables' nodes (150 to 640 K), against six Newton steps
on the table in numpy, and logexp.cuh's halving near the smallest numbers."""
import ctypes
import os
import shutil
import subprocess
import tempfile

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from conftest import ROOT

pytestmark = pytest.mark.gpu
RV = 8.314462618 / 0.018015
LN100 = np.log(100.0)
# Sonntag's ln p = a/T + b + c T + d T^2 + e ln T, over liquid and over ice, in Pa
CURVE = ((-6096.9385, 16.635794 + LN100, -2.711193e-2, 1.673952e-5, 2.433502),
         (-6024.5282, 24.7219 + LN100, 1.0613868e-2, -1.3198825e-5, -0.49382577))
NODES = 150.0 + 0.5 * np.arange(981)


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    so = os.path.join(tempfile.mkdtemp(), "fp64_edges_check.so")
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17", "--expt-relaxed-constexpr", "-shared",
                    "-Xcompiler", "-fPIC", "-o", so, os.path.join(ROOT, "tests", "kernels", "fp64_edges_check.cu")], check=True)
    L = ctypes.CDLL(so)
    L.fp64_edges.argtypes = [ctypes.c_int] + [ctypes.c_void_p] * 3 + [ctypes.c_int]
    tab = torch.tensor(np.stack([_table(0), _table(1), np.zeros((981, 3))]), device="cuda")   # the third property is not read

    def run(which, x):
        X = torch.tensor(np.asarray(x, dtype=np.float64), device="cuda")
        R = torch.empty_like(X)
        torch.cuda.synchronize()
        assert L.fp64_edges(which, X.data_ptr(), tab.data_ptr(), R.data_ptr(), X.numel()) == 0
        return R.cpu().numpy()

    return run


def _table(ice):
    a, b, c, d, e = CURVE[ice]
    T = NODES
    return np.stack([a / T + b + T * (c + T * d) + e * np.log(T), -a / T ** 2 + c + 2 * d * T + e / T,
                     0.5 * (2 * a / T ** 3 + 2 * d - e / T ** 2)], axis=1)


def _eval(tab, T):
    """Value, slope and the sum of the terms' magnitudes of the tabulated curve (end nodes extrapolate)."""
    k = np.clip(np.floor((T - 150.0) * 2 + 0.5), 0, 980).astype(int)
    d, (c0, c1, c2) = T - NODES[k], tab[k].T
    return c0 + d * (c1 + d * c2), c1 + 2 * c2 * d, np.abs(c0) + np.abs(d * c1) + d * d * np.abs(c2)


# Both sides solve the same equation; what may differ is the rounding of the curve's value (four
# operations on terms of the given size, on either side) over its slope, and of the root itself.
@pytest.mark.parametrize("ice", [0, 1])
def test_tabulated_saturation_temperature_beyond_the_nodes(lib, ice):
    tab = _table(ice)
    lnpv = np.concatenate([np.linspace(-69.0776, 16.5, 8000), [-69.07755278982137, -12.0, -11.0],
                           np.linspace(16.5, 20.0, 500) if not ice else []])   # the ice curve has its maximum near 17
    T = 1.0 / (1.0 / 273.15 - RV * (lnpv - np.log(611.2)) / (2.501e6 + (3.337e5 if ice else 0.0)))
    for _ in range(6):
        v, s, _ = _eval(tab, T)
        T = T - (v - lnpv) / s
    v, s, mag = _eval(tab, T)
    assert np.abs(v - lnpv).max() < 1e-12          # the oracle's root is one
    eps = 2.0 ** -52
    tol = 8 * eps * (mag + np.abs(lnpv)) / np.abs(s) + 4 * eps * np.abs(T)
    got = lib(ice, lnpv)
    bad = ~(np.abs(got - T) <= tol)
    assert not bad.any(), (lnpv[bad][:3], got[bad][:3], T[bad][:3])


# An exact half, rounded to even where a subnormal's last bit goes, as the multiplication by 1/2 is.
def test_halving_near_the_smallest_numbers(lib):
    g = np.random.default_rng(6)
    low = (g.integers(0, 1 << 54, 4000, dtype=np.uint64) >> g.integers(0, 54, 4000, dtype=np.uint64))   # below 2^-1020
    x = np.concatenate([low.view(np.float64), 5e-324 * np.arange(9), 2.0 ** np.arange(-1074.0, -1015.0),
                        [np.nextafter(2.0 ** -1021, 0), np.nextafter(2.0 ** -1022, 0), 1.7976931348623157e308, np.inf]])
    x = np.concatenate([x, -x])
    with np.errstate(under="ignore"):
        want = 0.5 * x
    got = lib(2, x)
    assert np.array_equal(got.view(np.int64), want.view(np.int64))
    assert np.isnan(lib(2, [np.nan])).all()
