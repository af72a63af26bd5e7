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



def test_ends_of_the_accepted_range(tmp_path):
    """States at the ends of what fix_state takes: beta = -q4/2 from 2^-80 up to (not
    including) 2^80, |q1| just below 32, |S|^2 up to 15.4. Against multiple precision
    at the bound of the flux tests; one step outside is left to the FP64 form."""
    mp = pytest.importorskip("mpmath")
    import test_fixed_flux as flux
    mp.mp.dps = 40
    out = str(tmp_path / "libfixed.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I" + CSRC, "-o", out,
                    os.path.join(HERE, "fixed_flux_shim.cpp")], check=True)
    so = ctypes.CDLL(out)

    def shim(qi, q0, nx, ny, along, sgn):
        n = len(nx)
        a = [np.ascontiguousarray(v, dtype=np.float64) for v in (qi, q0, nx, ny)]
        b = [np.ascontiguousarray(v, dtype=np.int32) for v in (along, sgn)]
        dG, ok = np.zeros((n, 4)), np.zeros(n, dtype=np.int32)
        so.fixed_flux(ctypes.c_long(n), *[_ptr(v) for v in a + b + [dG, ok]])
        return dG, ok.astype(bool)

    rng = np.random.default_rng(12)

    def states(beta, n):
        a, S = rng.uniform(0, 2 * np.pi, n), np.sqrt(rng.uniform(0, 15.4, n))
        q1 = rng.choice([-31.99, 31.99, 0.3], n) + 0.005 * rng.uniform(-1, 1, n)
        return np.stack([q1, 2 * S * np.cos(a) * np.sqrt(beta), 2 * S * np.sin(a) * np.sqrt(beta), -2 * beta], axis=-1)

    n = 96
    ends = [2.0 ** -80, np.nextafter(2.0 ** -79, 0), 2.0 ** -79 * 1.5, 2.0 ** 79, np.nextafter(2.0 ** 80, 0), 2.0 ** 78 * 1.25, 1.0]
    for beta in ends:
        q = states(np.full(n, beta), n)
        near = q * np.array([1, 1 + 1e-5, 1 - 1e-5, 1])
        flux._check(shim, q, near, rng)
    flux._check(shim, states(rng.choice(ends[:3], n), n), states(rng.choice(ends[3:6], n), n), rng)   # one state at each end
    good = states(np.ones(4), 4)
    one = np.ones(4)
    for beta in (np.nextafter(2.0 ** -80, 0), 2.0 ** 80):
        q = states(np.full(4, beta), 4)
        assert not shim(q, good, one, 0 * one, one, one)[1].any() and not shim(good, q, one, 0 * one, one, one)[1].any()
