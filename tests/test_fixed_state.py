"""What a state passes through on its way to the fixed-point fluxes
(csrc/lskum_fixed.cuh), compiled for the host, against exact rationals.
"""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2403_13287_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("state") / "libstate.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I" + CSRC, "-o", out,
                    os.path.join(HERE, "fixed_state_shim.cpp")], check=True)
    return ctypes.CDLL(out)


def _ptr(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def test_quotient_rounds_once(lib):
    """rho/p and 1/p: the reciprocal within 2^-60, the product within 1.25 units of
    2^-60 more, so 2^-53 (1 + 2^-4) relative to the exact quotient."""
    rng = np.random.default_rng(3)
    n = 4000
    a = np.exp(rng.uniform(-2, 2, (n, 2)))
    a[:500] = 2.0 ** rng.integers(-2, 3, (500, 2)) * (1 + rng.choice([0, 2.0 ** -52, -(2.0 ** -53), 2.0 ** -30], (500, 2)))
    a[500:1000] = 2.0 ** rng.uniform(-300, 300, (500, 2))
    r, q, ok = np.zeros(n), np.zeros(n), np.zeros(n, dtype=np.int32)
    lib.fixed_quotient(ctypes.c_long(n), _ptr(a), _ptr(r), _ptr(q), _ptr(ok))
    assert ok.all()
    for e in range(n):
        x, y = Fraction(float(a[e, 0])), Fraction(float(a[e, 1]))
        for got, want in ((r[e], 1 / y), (q[e], x / y)):
            assert abs(Fraction(float(got)) - want) <= want * Fraction(17, 16) / 2 ** 53
    bad = np.array([[0.0, 1], [1, 0.0], [-1, 1], [1, -1], [np.nan, 1], [1, np.inf], [1e-310, 1], [1, 1e300]])
    m = len(bad)
    r, q, ok = np.zeros(m), np.zeros(m), np.zeros(m, dtype=np.int32)
    lib.fixed_quotient(ctypes.c_long(m), _ptr(bad), _ptr(r), _ptr(q), _ptr(ok))
    assert not ok.any()

