"""The two polynomials of the integer-pipe sine and cosine on their own give the bits
of the joint evaluation, one the sine and the other the cosine (CPU build)."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2011_01740_gb300", "csrc")


def test_halves_give_the_joint_bits(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    so = str(tmp_path / "halves.so")
    subprocess.run([gxx, "-O2", "-std=c++17", "-shared", "-fPIC", f"-I{CSRC}",
                    os.path.join(HERE, "sincos_half_host.cpp"), "-o", so], check=True)
    rng = np.random.default_rng(5)
    eighths = np.arange(-16, 17) / 8
    x = np.concatenate([rng.uniform(-3, 3, 20000), np.exp(rng.uniform(-700, 200, 2000)), eighths,
                        np.nextafter(eighths, 9), np.nextafter(eighths, -9),
                        [0.0, -0.0, 5e-324, 2.0 ** 52, 2.0 ** 53 + 2, 1e300, np.inf, -np.inf, np.nan]])
    P = ctypes.POINTER(ctypes.c_double)
    both, halves = np.zeros((x.size, 2)), np.full((x.size, 2), 7.0)
    ctypes.CDLL(so).sincos_halves(ctypes.c_long(x.size), x.ctypes.data_as(P), both.ctypes.data_as(P), halves.ctypes.data_as(P))
    assert np.array_equal(both.view(np.int64), halves.view(np.int64))
