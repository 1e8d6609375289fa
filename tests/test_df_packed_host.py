"""The packed double-float operations (csrc/df.cuh, two values per instruction)
give both halves the bits of the scalar ones: cancelling, equal, tiny and large
operands, zeros of either sign."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2011_01740_gb300", "csrc")


@pytest.mark.parametrize("kind", ["random", "cancel", "special"])
def test_packed_halves_are_the_scalar_bits(tmp_path, kind):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    so = str(tmp_path / "packed.so")
    subprocess.run([gxx, "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", f"-I{CSRC}",
                    os.path.join(HERE, "df_packed_host.cpp"), "-o", so], check=True)
    rng = np.random.default_rng(1)
    if kind == "special":
        v = np.array([0.0, -0.0, 1.0, -1.0, 1.0 + 2.0**-40, 3e-25, -7e24])
        a, b = (x.ravel() for x in np.meshgrid(v, v))
    else:
        n = 100_000
        a = rng.normal(size=n) * 10.0 ** rng.uniform(-12, 12, n)
        b = rng.normal(size=n) * 10.0 ** rng.uniform(-12, 12, n)
        if kind == "cancel":
            b = -a * (1.0 + rng.integers(-3, 4, n) * 2.0 ** rng.integers(-50, -20, n).astype(float))
    a, b = np.ascontiguousarray(a), np.ascontiguousarray(b)
    out = np.zeros((a.size, 3, 2, 4), dtype=np.float32)
    P = ctypes.POINTER(ctypes.c_double)
    ctypes.CDLL(so).packed_ops(a.size, a.ctypes.data_as(P), b.ctypes.data_as(P),
                               out.ctypes.data_as(ctypes.POINTER(ctypes.c_float)))
    # equal as numbers: a zero's sign may differ (x - y is formed as a fused y (-1) + x)
    assert np.array_equal(out[:, :, 0], out[:, :, 1], equal_nan=True)   # (-7e24)^2 overflows in both
