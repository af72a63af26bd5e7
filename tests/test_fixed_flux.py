"""The fixed-point parts of the FP64 form (csrc/lskum_fixed.cuh): the split
fluxes, and the dot products, differences and limiter quotients of the
q-derivative passes.

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
from fractions import Fraction

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


def _rows(shim, name, a):
    out, ok = np.zeros(len(a)), np.zeros(len(a), dtype=np.int32)
    a = np.ascontiguousarray(a)
    getattr(shim.lib, name)(ctypes.c_long(len(a)), a.ctypes.data_as(ctypes.c_void_p), out.ctypes.data_as(ctypes.c_void_p),
                            ok.ctypes.data_as(ctypes.c_void_p))
    return out, ok.astype(bool)


@pytest.mark.parametrize("spread", [0, 30, 120])
def test_dot_products(shim, spread):
    """h . g against exact rationals: the products' dropped words cost at most
    2 units of 2^-58 |h||g| and the stored form of h 2^-57 of |h| (together
    below 2^-55.4), then one rounding."""
    rng = np.random.default_rng(5)
    n = 3000
    a = rng.standard_normal((n, 4)) * 2.0 ** rng.integers(-spread, spread + 1, (n, 4))
    a[:50, 1], a[50:100, 2], a[100:150, 3], a[150:200, 2:] = 0.0, 0.0, 0.0, 0.0
    a[200:400, 3] = -a[200:400, 0] * a[200:400, 2] / a[200:400, 1]     # cancelling sums
    c, ok = _rows(shim, "fixed_dot", a)
    assert ok[:150].all() and ok[200:].mean() > 0.9
    for e in np.nonzero(ok)[0]:
        h0, h1, g0, g1 = [Fraction(float(v)) for v in a[e]]
        exact = h0 * g0 + h1 * g1
        size = Fraction(float(np.hypot(a[e, 0], a[e, 1]))) * Fraction(float(np.hypot(a[e, 2], a[e, 3])))
        assert abs(Fraction(float(c[e])) - exact) <= abs(exact) / 2 ** 53 + size * Fraction(1, 2 ** 55)


def test_dot_product_range(shim):
    # a non-finite gradient or too extreme an exponent is left to FP64
    bad = [[1, 1, np.inf, 0], [1, 1, 0, np.nan], [1, 1, -np.inf, np.inf], [1e39, 1, 1, 1], [1e-39, 0, 1, 1],
           [1, 1, 1e308, 0], [1, 1, 5e-324, 0], [1, 1, 1e-300, 0], [0, 0, 1, 1]]
    assert not _rows(shim, "fixed_dot", np.array(bad, dtype=float))[1].any()


@pytest.mark.parametrize("eps,d", [(-60, -10), (-10, -30), (-20, -10), (-500, -200)])
def test_limiter_quotient(shim, eps, d):
    """f(x, d) relative to exact rationals: operands within 2^-59, three
    truncated products of order 2^-56 each over M >= 1/4, the reciprocal within
    2^-60: below 2^-53, then one rounding."""
    rng = np.random.default_rng(6)
    n = 2000
    D = rng.uniform(0.5, 2, n) * 2.0 ** rng.uniform(d - 5, d + 5, n)
    X = 2 * D * rng.uniform(0, 1, n)
    E = rng.uniform(0.5, 2, n) * 2.0 ** rng.uniform(eps - 10, eps + 10, n)
    X[:100] = 0.0
    E[100:200] = 0.0
    X[200:300] = np.nextafter(2 * D[200:300], 0)
    X[300:400] = D[300:400] * 2.0 ** rng.uniform(-60, -20, 100)
    f, ok = _rows(shim, "fixed_phi", np.stack([X, D, E], axis=1))
    assert ok.all() and np.all(f >= 0) and np.all(f <= 1)
    for e in range(n):
        x, dd, ep = Fraction(float(X[e])), Fraction(float(D[e])), Fraction(float(E[e]))
        want = (x * (x + 2 * dd) + ep) / (x * (x + dd) + 2 * dd * dd + ep)
        assert abs(Fraction(float(f[e])) - want) <= want * Fraction(2, 2 ** 53)


def test_logarithm_and_reciprocal(shim):
    """ln(rho) + 2.5 ln(beta) against multiple precision: each log2 within
    2 units of 2^-60, times 7/2 and 5/2, their sum cut to 2^-57 and a product
    within 1.25 units of 2^-56 (together below 2^-54), then one rounding; extreme
    exponents to two units in the last place. 1/rho: within 2^-59, then one rounding."""
    mp = pytest.importorskip("mpmath")
    mp.mp.dps = 40
    rng = np.random.default_rng(9)
    n = 1500
    a = np.exp(rng.uniform(-2, 2, (n, 2)))
    a[:300] = 2.0 ** rng.integers(-1, 2, (300, 2)) * (1 + rng.choice([0, 2.0 ** -52, -(2.0 ** -53), 1 / 1024, 1 / 2048], (300, 2)))
    a[300:500] = 2.0 ** rng.uniform(-300, 300, (200, 2))
    l, r, ok = np.zeros(n), np.zeros(n), np.zeros(n, dtype=np.int32)
    ptr = lambda v: v.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    shim.lib.fixed_log(ctypes.c_long(n), ptr(a), ptr(l), ptr(r), ptr(ok))
    assert ok.all()
    for e in range(n):
        rho, p = mp.mpf(float(a[e, 0])), mp.mpf(float(a[e, 1]))
        want = mp.log(rho) + mp.mpf(2.5) * mp.log(rho / (2 * p))
        assert abs(mp.mpf(float(l[e])) - want) <= mp.mpf(2) ** -54 + abs(want) * mp.mpf(2) ** (-51 if 300 <= e < 500 else -53)
        assert abs(mp.mpf(float(r[e])) * rho - 1) <= mp.mpf(2) ** -53 + mp.mpf(2) ** -58
    bad = np.array([[0.0, 1], [-1, 1], [np.inf, 1], [np.nan, 1], [1, 0], [1, -0.0], [1, np.nan], [1e-310, 1], [1e300, 1]])
    m = len(bad)
    l, r, ok = np.zeros(m), np.zeros(m), np.zeros(m, dtype=np.int32)
    shim.lib.fixed_log(ctypes.c_long(m), ptr(bad), ptr(l), ptr(r), ptr(ok))
    assert not ok.any()


def test_differences_are_exact(shim):
    rng = np.random.default_rng(7)
    a = rng.uniform(-4, 4, 4000)
    b = np.concatenate([a[:2000] * (1 + 1e-3 * rng.uniform(-1, 1, 2000)), rng.uniform(-4, 4, 2000)])
    b[:20] = a[:20]
    d, ok = _rows(shim, "fixed_difference", np.stack([a, b], axis=1))
    assert np.array_equal(ok, (np.signbit(a) == np.signbit(b)) & (np.frexp(a)[1] == np.frexp(b)[1]))
    assert np.array_equal(d[ok], (a - b)[ok]) and not np.signbit(d[:20]).any()
    special = np.array([[np.inf, np.inf], [np.nan, np.nan], [0.0, 0.0], [1e-310, 1e-310]])
    assert not _rows(shim, "fixed_difference", special)[1].any()


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


@pytest.mark.gpu
@pytest.mark.parametrize("order,limiter,boundary", [(1, 0.0, 0), (2, 0.0, 0), (2, 1.0, 0), (2, 1.0, 1)])
def test_every_launch_form_gives_the_same_bits(order, limiter, boundary):
    """The FP64 kernels split a point over more lanes the smaller the cloud: 4,
    2 or 1 pairs in the flux kernel, 4 or 2 lanes in the q-derivative passes.
    A 3250-point cloud alone, beside 18k points and beside 114k points in one
    batch (all three forms): bitwise the same states and residuals, and the
    18k cloud's residual at the oracle's bar."""
    import torch

    import oracle
    from paper_2403_13287_gb300.cloudgen import naca0012_cloud, smooth_state
    from paper_2403_13287_gb300.lskum import Solver
    a, mid, big = naca0012_cloud(130, 24, seed=11), naca0012_cloud(180, 99, seed=3, shuffle=True), naca0012_cloud(512, 221, seed=4)
    kw = dict(order=order, inner_iters=3, time_scheme=1, limiter_K=limiter, precision=0, reorder=1, boundary=boundary)
    U0 = {id(c): smooth_state(c, 0.85, 1.0, amp=0.05, seed=9) for c in (a, mid, big)}
    got = []
    for clouds in ([a], [a, mid], [a, mid, big], [mid]):
        if len(clouds) > 1:
            s = Solver.batch([(c, 0.85, 1.0) for c in clouds], **kw)
        else:
            s = Solver(clouds[0], mach=0.85, aoa_deg=1.0, **kw)
        U = np.ascontiguousarray(np.concatenate([U0[id(c)] for c in clouds], axis=1))
        R = s.residual(torch.from_numpy(U).cuda()).cpu().numpy()
        s.set_state(U)
        s.step(2)
        got.append((R, s.get_state()))
        s.close()
    n, m = a["n"], mid["n"]
    for R, V in got[1:3]:
        assert np.array_equal(R[:, :n], got[0][0]) and np.array_equal(V[:, :n], got[0][1])
        assert np.array_equal(R[:, n:n + m], got[3][0]) and np.array_equal(V[:, n:n + m], got[3][1])
    Ro, S = oracle.residual(mid, oracle.split_stencils(mid), U0[id(mid)], order=order, inner=3, limiter=limiter,
                            want_scale=True, boundary=boundary, mach=0.85, aoa_deg=1.0)
    assert np.all(np.abs(got[3][0] - Ro) <= 1e-12 * S + 1e-300)


@pytest.mark.gpu
@pytest.mark.parametrize("gamma,mach", [(1.4, 7.0), (1.3, 2.0)])
def test_vjp_across_the_range_matches_the_oracle(gamma, mach):
    """The two-lane flux adjoint with states on both sides of the fixed-point
    range, and the one-lane FP64 one (gamma = 1.3): sampled entries against
    complex-step derivatives, at the VJP tests' 1e-10 of the largest."""
    import torch

    import oracle
    from oracle import lskum_jvp
    from paper_2403_13287_gb300.cloudgen import naca0012_cloud
    from paper_2403_13287_gb300.lskum import Solver
    c = naca0012_cloud(130, 24, seed=11)
    rng = np.random.default_rng(4)
    n = c["n"]
    rho, p = 1 + 0.2 * rng.uniform(-1, 1, n), (1 + 0.2 * rng.uniform(-1, 1, n)) / gamma
    m, a = mach * rng.uniform(0, 1, n), rng.uniform(0, 2 * np.pi, n)
    u, v = m * np.sqrt(gamma * p / rho) * np.cos(a), m * np.sqrt(gamma * p / rho) * np.sin(a)
    U = np.ascontiguousarray(np.stack([rho, rho * u, rho * v, p / (gamma - 1) + 0.5 * rho * (u * u + v * v)]))
    Rb = rng.standard_normal((4, n))
    s = Solver(c, order=1, inner_iters=0, mach=0.8, aoa_deg=1.0, gamma=gamma, reorder=1)
    Ub, xb, yb = (t.cpu().numpy() for t in s.residual_vjp(torch.from_numpy(Rb).cuda(), torch.from_numpy(U).cuda()))
    s.close()
    ent = [("U", int(rng.integers(4)), int(k)) for k in rng.choice(n, 40, replace=False)]
    ent += [(d, int(k)) for d in "xy" for k in rng.choice(n, 20, replace=False)]
    want = lskum_jvp.vjp_entries(c, oracle.split_stencils(c), U, Rb, ent, order=1, inner=0, gamma=gamma)
    got = np.array([Ub[e[1], e[2]] if e[0] == "U" else (xb if e[0] == "x" else yb)[e[1]] for e in ent])
    for kind in "Uxy":
        k = [i for i, e in enumerate(ent) if e[0] == kind]
        assert np.all(np.abs(got - want)[k] <= 1e-10 * np.abs(want).max())


@pytest.mark.gpu
@pytest.mark.parametrize("precision,fp32,limiter", [(0, False, 0.0), (0, False, 1.0), (1, True, 0.0)])
def test_state_cotangent_alone_is_that_of_the_full_product(precision, fp32, limiter):
    """Without coordinate cotangents the reverse pass skips the weights' and
    offsets' ones: U_bar is the same. (FP64 bitwise; FP32 to 1e-6 of its
    largest entry: the two instantiations may contract differently.)"""
    import torch

    from paper_2403_13287_gb300.cloudgen import naca0012_cloud, smooth_state
    from paper_2403_13287_gb300.lskum import Solver
    c = naca0012_cloud(180, 99, seed=3, shuffle=True)
    U = torch.from_numpy(smooth_state(c, 0.85, 1.0, amp=0.05, seed=9)).cuda()
    Rb = torch.from_numpy(np.random.default_rng(1).standard_normal((4, c["n"]))).cuda()
    s = Solver(c, order=2, inner_iters=3, limiter_K=limiter, precision=precision, reorder=1)
    full = s.residual_vjp(Rb, U, fp32=fp32)[0].cpu().numpy()
    only = s.residual_vjp(Rb, U, want_xy=False, fp32=fp32)[0].cpu().numpy()
    s.close()
    if fp32:
        assert np.abs(full - only).max() <= 1e-6 * np.abs(full).max()
    else:
        assert np.array_equal(full, only)


@pytest.mark.gpu
@pytest.mark.parametrize("W,L,K", [(34, 12, 1.0), (50, 14, 0.3)])
def test_limited_vjp_at_the_last_points_matches_the_oracle(W, L, K):
    """The limiter's reverse takes four lanes per point: clouds that end inside
    a warp, entries at the last points and the wall, against complex-step
    derivatives at the VJP tests' 1e-10 of the largest."""
    import torch

    import oracle
    from oracle import lskum_jvp
    from paper_2403_13287_gb300.cloudgen import naca0012_cloud, smooth_state
    from paper_2403_13287_gb300.lskum import Solver
    c = naca0012_cloud(W, L, seed=5)
    n = c["n"]
    assert n % 32 and n % 8
    rng = np.random.default_rng(W)
    U = smooth_state(c, 0.85, 1.0, amp=0.05, seed=4)
    Rb = rng.standard_normal((4, n))
    s = Solver(c, order=2, inner_iters=2, mach=0.85, aoa_deg=1.0, limiter_K=K, reorder=0)
    Ub, xb, yb = (t.cpu().numpy() for t in s.residual_vjp(torch.from_numpy(Rb).cuda(), torch.from_numpy(U).cuda()))
    s.close()
    pts = list(range(n - 8, n)) + [int(k) for k in rng.choice(n - 8, 8, replace=False)]
    ent = [("U", int(rng.integers(4)), k) for k in pts] + [(d, k) for d in "xy" for k in pts]
    want = lskum_jvp.vjp_entries(c, oracle.split_stencils(c), U, Rb, ent, order=2, inner=2, limiter=K)
    got = np.array([Ub[e[1], e[2]] if e[0] == "U" else (xb if e[0] == "x" else yb)[e[1]] for e in ent])
    assert np.all(np.abs(got - want) <= 1e-10 * np.abs(want).max())


@pytest.mark.gpu
def test_the_sign_of_zero_does_not_matter_to_the_limiter_reverse():
    """The search for the extreme neighbours orders bit patterns: momenta of
    +0 and -0 are the same state and give the same cotangents."""
    import torch

    from paper_2403_13287_gb300.cloudgen import naca0012_cloud, smooth_state
    from paper_2403_13287_gb300.lskum import Solver
    c = naca0012_cloud(50, 14, seed=5)
    rng = np.random.default_rng(0)
    U = smooth_state(c, 0.85, 1.0, amp=0.05, seed=4)
    U[3] -= 0.5 * U[2] ** 2 / U[0]
    U[2] = 0.0
    Rb = torch.from_numpy(rng.standard_normal((4, c["n"]))).cuda()
    V = U.copy()
    V[2] = np.where(rng.random(c["n"]) < 0.5, -0.0, 0.0)
    s = Solver(c, order=2, inner_iters=2, mach=0.85, aoa_deg=1.0, limiter_K=1.0)
    a, b = (s.residual_vjp(Rb, torch.from_numpy(x).cuda()) for x in (U, V))
    s.close()
    for p, q in zip(a, b):
        assert torch.equal(p, q)


@pytest.mark.gpu
@pytest.mark.parametrize("limiter", [0.0, 1.0])
def test_both_lane_forms_of_the_reverse_gradient_passes(limiter):
    """One or two lanes per point by the size of the cloud: a 3250-point cloud
    alone and beside 64k points in one batch. U_bar bitwise; x_bar and y_bar,
    whose sums take their four terms in another order, to 1e-13 of the largest
    (2^-53 per addition of at most 20 edges' terms that cancel by up to 10)."""
    import torch

    from paper_2403_13287_gb300.cloudgen import naca0012_cloud, smooth_state
    from paper_2403_13287_gb300.lskum import Solver
    a, big = naca0012_cloud(130, 24, seed=11), naca0012_cloud(324, 197, seed=4)
    n = a["n"]
    kw = dict(order=2, inner_iters=3, time_scheme=1, limiter_K=limiter, precision=0, reorder=1)
    U0 = [smooth_state(c, 0.85, 1.0, amp=0.05, seed=9) for c in (a, big)]
    Rb = np.random.default_rng(2).standard_normal((4, n + big["n"]))
    got = []
    for clouds in ([a], [a, big]):
        m = sum(c["n"] for c in clouds)
        s = Solver.batch([(c, 0.85, 1.0) for c in clouds], **kw) if len(clouds) > 1 else Solver(a, mach=0.85, aoa_deg=1.0, **kw)
        U = np.ascontiguousarray(np.concatenate(U0[:len(clouds)], axis=1))
        out = s.residual_vjp(torch.from_numpy(np.ascontiguousarray(Rb[:, :m])).cuda(), torch.from_numpy(U).cuda())
        only = s.residual_vjp(torch.from_numpy(np.ascontiguousarray(Rb[:, :m])).cuda(), torch.from_numpy(U).cuda(), want_xy=False)[0]
        assert torch.equal(out[0], only)
        got.append([t.cpu().numpy()[..., :n] for t in out])
        s.close()
    assert np.array_equal(got[0][0], got[1][0])
    for p, q in zip(got[0][1:], got[1][1:]):
        assert np.abs(p - q).max() <= 1e-13 * np.abs(p).max()
