"""Host check of v / 4 by the exponent (csrc/pfc_fixed.cuh): the bits of 0.25 * v
wherever that is exact and normal, and for zeros, infinities and NaN; a zero of
v's sign below 2^-1020."""

import ctypes
import os
import shutil
import struct
import subprocess

import numpy as np
import pytest

HEADER_DIR = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                          "paper_1611_06288_gb300", "csrc")
SRC = '#include "pfc_fixed.cuh"\nextern "C" double quarter(double v) { return pfc::fix_quarter(v); }\n'


def bits(v):
    return struct.pack("<d", v)


def test_quarter_is_exact(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    (tmp_path / "q.cpp").write_text(SRC)
    so = tmp_path / "q.so"
    subprocess.run([gxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-I", HEADER_DIR,
                    str(tmp_path / "q.cpp"), "-o", str(so)], check=True)
    quarter = ctypes.CDLL(str(so)).quarter
    quarter.restype, quarter.argtypes = ctypes.c_double, [ctypes.c_double]
    rng = np.random.default_rng(4)
    vs = [0.0, np.inf, 1.0, 2.0 ** -1020, np.nextafter(2.0 ** -1019, 0), np.finfo(float).max]
    vs += list(rng.standard_normal(200) * 10.0 ** rng.uniform(-300, 300, 200))
    for v in vs:
        for s in (v, -v):
            assert bits(quarter(s)) == bits(0.25 * s), s
    assert np.isnan(quarter(np.nan))
    for v in (np.nextafter(2.0 ** -1020, 0), 5e-324, -5e-324):
        assert bits(quarter(v)) == bits(np.copysign(0.0, v))
