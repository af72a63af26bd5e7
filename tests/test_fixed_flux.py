"""The fixed-point split fluxes of the FP64 form (csrc/lskum_fixed.cuh).

CPU: the header compiled for the host against multiple precision, over the
range of states it accepts and at that range's edges, and the states it has to
leave to the FP64 form. GPU: residuals of clouds whose states straddle the
range (both forms in one warp) against the FP64 oracle.

Tolerance of the CPU test. The formats keep at least 54 bits of the factors
(rho r, rho r^2, rho r^3: relative error below 2^-53) and 2^-54.5 absolute of
the exponent's argument, so each flux carries below 2^-52 relative to its
natural scale rho r^j (1 + |S|)^j (twice that for the energy, whose enthalpy
is 1.75 + |S|^2/2), plus 2^-55 of it from the last product: 4 units of 2^-53
of the two states' summed scales bound the difference, rounded once more.
"""
import ctypes
import os
import re
import subprocess
import sys

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2403_13287_gb300", "csrc")


@pytest.fixture(scope="module")
def shim(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("fixed") / "libfixed.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I" + CSRC, "-o", out,
                    os.path.join(HERE, "fixed_flux_shim.cpp")], check=True)
    lib = ctypes.CDLL(out)

    def call(qi, q0, nx, ny, along, sgn):
        n = len(nx)
        a = [np.ascontiguousarray(v, dtype=np.float64) for v in (qi, q0, nx, ny)]
        b = [np.ascontiguousarray(v, dtype=np.int32) for v in (along, sgn)]
        dG, ok = np.zeros((n, 4)), np.zeros(n, dtype=np.int32)
        p = [v.ctypes.data_as(ctypes.c_void_p) for v in a + b + [dG, ok]]
        lib.fixed_flux(ctypes.c_long(n), *p)
        return dG, ok.astype(bool)

    call.lib = lib
    return call


def _q(rho, u, v, p):
    b = 0.5 * rho / p
    return np.stack([np.log(rho) + 2.5 * np.log(b) - b * (u * u + v * v), 2 * b * u, 2 * b * v, -2 * b], axis=-1)


def _flux(mp, q, nx, ny, along, sgn):
    """Split flux in multiple precision and the natural scales of its components."""
    q = [mp.mpf(float(c)) for c in q]
    nx, ny = mp.mpf(float(nx)), mp.mpf(float(ny))
    b = -q[3] / 2
    us, un = (q[1] * ny - q[2] * nx) / (2 * b), (q[1] * nx + q[2] * ny) / (2 * b)
    w2 = us * us + un * un
    rho = mp.exp(q[0] + b * w2) * b ** mp.mpf(-2.5)
    p, (d, t) = rho / (2 * b), ((us, un) if along else (un, us))
    S = d * mp.sqrt(b)
    A, B = (1 + sgn * mp.erf(S)) / 2, sgn * mp.exp(-S * S) / (2 * mp.sqrt(mp.pi * b))
    E, m = p * mp.mpf(2.5) + rho * w2 / 2, rho * (d * A + B)
    r, k = 1 / mp.sqrt(b), 1 + mp.sqrt(b * w2)
    return ([m, (p + rho * d * d) * A + rho * d * B, t * m, (E + p) * d * A + (E + p / 2) * B],
            [rho * r * k, rho * (r * k) ** 2, rho * (r * k) ** 2, 2 * rho * (r * k) ** 3])


def _check(shim, q0, qi, rng):
    mp = pytest.importorskip("mpmath")
    mp.mp.dps = 40
    n = len(q0)
    th = rng.uniform(0.0, 2.0 * np.pi, n)
    th[: n // 8] = rng.integers(0, 4, n // 8) * (np.pi / 2)      # axis-aligned frames
    nx, ny = np.cos(th), np.sin(th)
    along, sgn = rng.integers(0, 2, n), 2 * rng.integers(0, 2, n) - 1
    dG, ok = shim(qi, q0, nx, ny, along, sgn)
    assert ok.all()
    for e in range(n):
        a, sa = _flux(mp, qi[e], nx[e], ny[e], int(along[e]), int(sgn[e]))
        b, sb = _flux(mp, q0[e], nx[e], ny[e], int(along[e]), int(sgn[e]))
        for k in range(4):
            exact = a[k] - b[k]
            err = abs(exact - mp.mpf(float(dG[e, k])))
            assert err <= mp.mpf(2) ** -53 * (4 * (sa[k] + sb[k]) + abs(exact)), (e, k, float(err / (sa[k] + sb[k])))


# (largest Mach number, relative difference of the two states, density scale, pressure scale)
@pytest.mark.parametrize("mach,amp,rho,p", [(0.01, 0.05, 1.0, 1.0), (0.9, 1e-9, 1.0, 1.0), (2.0, 0.3, 1.0, 1.0),
                                           (3.4, 0.02, 1.0, 1.0), (0.3, 0.9, 1e3, 1e2), (1.2, 0.05, 1e-3, 1e-4),
                                           (1.0, 0.05, 1e-2, 1e2), (1.0, 0.05, 1e2, 1e-2)])
def test_fixed_flux_matches_multiple_precision(shim, mach, amp, rho, p):
    rng = np.random.default_rng(7)
    n = 160
    r = rho * (1 + 0.3 * rng.uniform(-1, 1, n))
    pr = p / 1.4 * (1 + 0.3 * rng.uniform(-1, 1, n))
    m, a = mach * np.sqrt(rng.uniform(0, 1, n)), rng.uniform(0, 2 * np.pi, n)
    c = np.sqrt(1.4 * pr / r)
    u, v = m * c * np.cos(a), m * c * np.sin(a)
    f = [1 + amp * rng.uniform(-1, 1, n) for _ in range(4)]
    _check(shim, _q(r, u, v, pr), _q(r * f[0], u * f[1], v * f[2], pr * f[3]), rng)


def test_range_and_zero_velocity(shim):
    rng = np.random.default_rng(8)
    n = 64
    # |S|^2 < 15.5 (= 3.9375^2, the bound on each component before the turn into the frame) is taken, above 15.875 not
    for S2, taken in ((15.49, True), (15.88, False)):
        a = rng.uniform(0, 2 * np.pi, n)
        S = np.sqrt(S2)
        q = _q(np.ones(n), np.sqrt(2.0) * S * np.cos(a), np.sqrt(2.0) * S * np.sin(a), np.ones(n))
        if taken:
            _check(shim, q, q * (1 - 1e-4), rng)
        else:
            assert not shim(q, q, np.ones(n), np.zeros(n), np.ones(n), np.ones(n))[1].any()
    # gas at rest, one momentum zero, and equal states (difference exactly zero)
    z = np.zeros(n)
    q = _q(1 + 0.1 * rng.uniform(-1, 1, n), z, z, np.ones(n))
    _check(shim, q, _q(np.ones(n), 0.3 * np.ones(n), z, np.ones(n)), rng)
    assert not shim(q, q, np.ones(n), z, np.ones(n), np.ones(n))[0].any()
    # what is not a state, or is too extreme: zero, positive, infinite and NaN q4, NaN elsewhere, huge q1
    bad = [[0, 0, 0, 0.0], [0, 0, 0, -0.0], [0, 0, 0, 1.0], [0, 0, 0, -np.inf], [0, 0, 0, np.nan], [np.nan, 0, 0, -2.0],
           [0, np.nan, 0, -2.0], [0, 0, np.inf, -2.0], [33.0, 0, 0, -2.0], [-np.inf, 0, 0, -2.0], [0, 1e300, 0, -2.0],
           [0, 0, 0, -1e-300], [0, 0, 0, -1e300], [0, 0, 0, -5e-324]]
    good = np.tile(_q(np.ones(1), 0.5 * np.ones(1), z[:1], np.ones(1)), (len(bad), 1))
    one, zero = np.ones(len(bad)), np.zeros(len(bad))
    assert not shim(np.array(bad, dtype=float), good, one, zero, one, one)[1].any()
    assert not shim(good, np.array(bad, dtype=float), one, zero, one, one)[1].any()


def test_words_at_the_ends_of_their_ranges(shim):
    """Operands whose low word rounds the high word up, at the largest values
    the formats meet (random states reach them once in 2^31): the table
    argument just below the middle between grid points (u just below 1), the
    exponent's remainder likewise, and factors with all bits set."""
    mp = pytest.importorskip("mpmath")
    mp.mp.dps = 40
    ll = lambda v: np.array(v, dtype=np.int64)  # noqa: E731
    ptr = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    # S = (k + 1/2) 2^-11 -+ a few units of 2^-61, both signs
    mid = [(k << 50) + (1 << 49) + d for k in (0, 1, 777, 2048, 8158) for d in (-(1 << 17), -(1 << 16) - 1, -3, -1, 0, 1)]
    S = ll(mid + [-v for v in mid])
    So, H = ll([3 << 59] * len(S)), ll([(7 << 57) + (1 << 58)] * len(S))
    F = np.zeros((len(S), 4), dtype=np.int64)
    shim.lib.fixed_parts(ctypes.c_long(len(S)), ptr(S), ptr(So), ptr(H), ptr(F))
    for e, v in enumerate(S):
        z = mp.ldexp(mp.mpf(int(v)), -61)
        Phi, E = (1 + mp.erf(z)) / 2, mp.exp(-z * z) / (2 * mp.sqrt(mp.pi))
        P = z * Phi + E
        want = [P, Phi / 2 + z * P, mp.mpf(0.75) * P, 2 * mp.mpf(1.125) * P - E / 4]
        for k, (w, q) in enumerate(zip(want, (61, 58, 58, 57))):
            # T and E within 2^-55.5 (the 32-bit coefficients), times |z| < 4 and H < 10
            assert abs(w - mp.ldexp(mp.mpf(int(F[e, k])), -q)) < mp.mpf(2) ** -53 * (1 + z * z), (e, k)
    # x log2(e) just below the middle between multiples of 1/4096
    log2e = 1 / mp.log(2)
    x = []
    for n in (-30 * 4096 - 5, -1, 0, 17, 4095, 20 * 4096 + 9):
        c = int((mp.mpf(n) + mp.mpf(1) / 2) / 4096 / log2e * mp.mpf(2) ** 57)
        x += [c + d for d in range(-4, 5)]
    x, M, m = ll(x), np.zeros(len(x), dtype=np.int64), np.zeros(len(x), dtype=np.int32)
    shim.lib.fixed_exp(ctypes.c_long(len(x)), ptr(x), ptr(M), ptr(m))
    for e, v in enumerate(x):
        w = mp.exp(mp.ldexp(mp.mpf(int(v)), -57))
        got = mp.ldexp(mp.mpf(int(M[e])), int(m[e]) - 62)
        # the log2 in Q55 within 1.25 units and the constant's 2^-63 of |x| < 32
        assert abs(got / w - 1) < mp.mpf(2) ** -54 and 0.9999 * 2 ** 62 < int(M[e]) < 2 ** 63 - 2 ** 31
    # factors of all bits set, and of the low word's top bit set
    c = ll([(1 << b) - d for b in (55, 58, 60, 61, 62) for d in (1, 2, 1 << 20, (1 << 31) - 1)])
    one = ll([1 << 54] * len(c))
    Fs = ll([(1 << 62) - 1] * len(c))
    gi, g0, ex = np.zeros_like(c), np.zeros_like(c), np.zeros(len(c), dtype=np.int32)
    shim.lib.fixed_scaled(ctypes.c_long(len(c)), ptr(c), ptr(one), ptr(Fs), ptr(gi), ptr(g0), ptr(ex))
    for e in range(len(c)):
        for got, fac in ((gi[e], int(c[e])), (g0[e], 1 << 54)):
            assert abs(mp.ldexp(mp.mpf(int(got)), int(ex[e])) - mp.mpf(fac) * int(Fs[e]) / mp.mpf(2) ** 64) <= mp.ldexp(mp.mpf(1.25), int(ex[e])), e


def test_tables_are_the_generator_output(tmp_path):
    pytest.importorskip("mpmath")
    work = tmp_path / "csrc"
    work.mkdir()
    (work / "gen_fix_tables.py").write_text(open(os.path.join(CSRC, "gen_fix_tables.py")).read())
    subprocess.run([sys.executable, str(work / "gen_fix_tables.py")], check=True)
    text = open(os.path.join(CSRC, "fix_tables.h")).read()
    assert (work / "fix_tables.h").read_text() == text
    # the last row an accepted state can reach: sqrt(15.875) 2048 = 8160
    assert int(re.search(r"#define LSKUM_FIX_KMAX (\d+)", text).group(1)) >= 8161


@pytest.mark.gpu
@pytest.mark.parametrize("boundary", [0, 1])
@pytest.mark.parametrize("gamma,mach", [(1.4, 7.0), (1.4, 2.0), (1.3, 2.0)])
def test_residual_across_the_range_matches_the_oracle(gamma, mach, boundary):
    """First-order residual of random states up to `mach` at every point: at
    Mach 7 many members leave the fixed-point range; gamma = 1.3 takes the
    FP64 form throughout. The FP64 bar of the parity tests, 1e-12 of the
    summand scale."""
    import torch

    import oracle
    from paper_2403_13287_gb300.cloudgen import naca0012_cloud
    from paper_2403_13287_gb300.lskum import Solver
    c = naca0012_cloud(130, 24, seed=11)
    rng = np.random.default_rng(4)
    n = c["n"]
    rho, p = 1 + 0.2 * rng.uniform(-1, 1, n), (1 + 0.2 * rng.uniform(-1, 1, n)) / gamma
    m, a = mach * rng.uniform(0, 1, n), rng.uniform(0, 2 * np.pi, n)
    u, v = m * np.sqrt(gamma * p / rho) * np.cos(a), m * np.sqrt(gamma * p / rho) * np.sin(a)
    U = np.ascontiguousarray(np.stack([rho, rho * u, rho * v, p / (gamma - 1) + 0.5 * rho * (u * u + v * v)]))
    s = Solver(c, order=1, inner_iters=0, mach=0.8, aoa_deg=1.0, gamma=gamma, reorder=1, boundary=boundary)
    R = s.residual(torch.from_numpy(U).cuda()).cpu().numpy()
    s.close()
    Ro, S = oracle.residual(c, oracle.split_stencils(c), U, order=1, inner=0, gamma=gamma, want_scale=True,
                            boundary=boundary, mach=0.8, aoa_deg=1.0)
    err = np.abs(R - Ro) / np.maximum(S, 1e-300)
    assert np.all(np.abs(R - Ro) <= 1e-12 * S), err.max()
