"""The branch-free square root, quotient, reciprocal and 2^x of surrogate.cuh
against CUDA's general forms, bit for bit, over every binary32 argument that the
features and the training pass them (the quotient over many cut-offs)."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1908_11118_gb300 import build as B

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def differences(tmp_path_factory):
    here = os.path.dirname(os.path.abspath(__file__))
    so = str(tmp_path_factory.mktemp("math") / "feature_math.so")
    cmd = [B.nvcc(), *B.ARCH, *B.FLAGS, "-I", B.CSRC, "-shared", "-o", so, os.path.join(here, "feature_math.cu")]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    f = ctypes.CDLL(so).feature_math_differences
    f.restype = ctypes.c_longlong
    f.argtypes = [ctypes.c_int, ctypes.c_float, ctypes.c_float, ctypes.c_void_p, ctypes.c_int]

    def run(what, lo, hi, divisors=(1.0,)):
        d = np.asarray(divisors, np.float32)
        return f(what, lo, hi, d.ctypes.data_as(ctypes.c_void_p), len(d))

    return run


def test_root(differences):
    assert differences(0, 1e-30, 2.0 ** 60) == 0


def test_quotient(differences):
    """Arguments up to pi rc: cut-offs in use, spread over twelve decades, and with
    the least and the largest mantissas."""
    rng = np.random.default_rng(5)
    rc = np.concatenate([[2.5, 2.9, 3.0, 4.775, 1.9375], rng.uniform(0.5, 20.0, 150), 10.0 ** rng.uniform(-6, 6, 60),
                         np.nextafter(np.float32([1, 2, 4, 8]), np.float32(0)),
                         np.nextafter(np.float32([1, 2, 4, 8]), np.float32(9))]).astype(np.float32)
    assert differences(1, 1e-15, 2.0 ** 40, rc) == 0


def test_reciprocal(differences):
    assert differences(2, 1.0, 2.0 ** 117) == 0


@pytest.mark.parametrize("what", [3, 4])   # 2^x, 2^-x
def test_exponential(differences, what):
    assert differences(what, 1e-30, 126.0) == 0


def test_a_difference_is_counted(differences):
    """Beyond the range in use 2^-x is a subnormal number, which the short form drops:
    every argument from 127 to 140 differs."""
    lo, hi = np.array([127.0, 140.0], np.float32).view(np.int32)
    assert differences(4, 127.0, 140.0) == hi - lo
