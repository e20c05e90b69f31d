"""Every entry of logexp_tables.cuh, made anew with mpmath at 200 bits."""
import os
import re

import numpy as np
import pytest

mp = pytest.importorskip("mpmath")

from conftest import ROOT


@pytest.fixture(scope="module")
def text():
    with open(os.path.join(ROOT, "paper_2504_20742_gb300", "csrc", "logexp_tables.cuh")) as fh:
        return fh.read()


def _array(text, name):
    body = re.search(name + r"\[\d+\] = \{(.*?)\}", text, re.S).group(1)
    return [v.strip() for v in body.split(",") if v.strip()]


def _constant(text, name):
    return re.search(name + r" = ([^;]+);", text).group(1)


def _f32(v):
    return np.float32(v.rstrip("f"))


def _hi_lo():
    """(hi, lo) of the logarithms, of the powers, of ln 2 and of ln2 / 512."""
    with mp.workprec(200):
        at42 = lambda v: mp.nint(v * 2 ** 42) / mp.mpf(2) ** 42
        logs = [-mp.log(mp.mpf(k) / 1024) for k in range(512, 1025)]
        pows = [mp.mpf(2) ** (mp.mpf(i) / 512) for i in range(512)]
        ln2 = mp.log(2)
        split = lambda v, h: (float(h), float(v - h))
        powers = [(float(v), float((v - mp.mpf(float(v))) / v)) for v in pows]
        return [split(v, at42(v)) for v in logs], powers, split(ln2, at42(ln2)), split(ln2 / 512, mp.mpf(float(ln2 / 512)))


def test_every_entry(text):
    logs, pows, ln2, l512 = _hi_lo()
    for hi, lo, want in (("LOG_HI", "LOG_LO", logs), ("EXP_HI", "EXP_LO", pows)):
        assert [float.fromhex(v) for v in _array(text, hi)] == [h for h, _ in want]
        assert [_f32(v) for v in _array(text, lo)] == [np.float32(v) for _, v in want]
    for name, (h, l) in (("LN2", ln2), ("L512", l512)):
        assert float.fromhex(_constant(text, name + "_H")) == h
        assert _f32(_constant(text, name + "_L")) == np.float32(l)
