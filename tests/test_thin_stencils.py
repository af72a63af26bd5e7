"""Two-term products h . grad q and a . g_bar where one direction's spacing is
far below the other's: a stencil stretched A : 1 along the axes, with the
gradient across its thin direction, has two terms of one size although |h||g|
is A times as large. The error counts against the terms.

CPU: the fixed-point product (csrc/lskum_fixed.cuh) against exact rationals.
GPU: q-derivatives of axis-aligned stretched clouds against extended
precision, and residual products against the complex-step oracle.
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
def dot(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("thin") / "libfixed.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I" + CSRC, "-o", out,
                    os.path.join(HERE, "fixed_flux_shim.cpp")], check=True)
    lib = ctypes.CDLL(out)

    def call(a):
        a = np.ascontiguousarray(a, dtype=np.float64)
        c, ok = np.zeros(len(a)), np.zeros(len(a), dtype=np.int32)
        lib.fixed_dot(ctypes.c_long(len(a)), *[v.ctypes.data_as(ctypes.c_void_p) for v in (a, c, ok)])
        return c, ok.astype(bool)

    return call


@pytest.mark.parametrize("cancel", [False, True])
@pytest.mark.parametrize("stretch", [0, 3, 10, 20, 40, 100])
def test_the_error_counts_against_the_terms(dot, stretch, cancel):
    """h = (1, 2^-s), grad q = (1, 2^s) times random factors. Each product loses at
    most 1.25 units of 2^-58 of itself and the alignment one unit more of the larger
    one: below 2^-56 of the two terms' sizes (3.5 units of 2^-58 of the larger), then
    one rounding of the sum."""
    rng = np.random.default_rng(stretch)
    n = 3000
    a = rng.uniform(0.5, 2.0, (n, 4)) * rng.choice([-1.0, 1.0], (n, 4))
    a[:, 1] *= 2.0 ** -stretch
    a[:, 3] *= 2.0 ** stretch
    a[n // 2:, 2] *= 2.0 ** rng.integers(-30, 31, n - n // 2)   # one term below the other
    a[:60, 0], a[60:120, 1], a[120:180, 2], a[180:240, 3] = 0.0, 0.0, 0.0, 0.0
    if cancel:
        a[240:, 3] = -a[240:, 0] * a[240:, 2] / a[240:, 1]
    c, ok = dot(a)
    assert ok.all()
    for e in range(n):
        h0, h1, g0, g1 = [Fraction(float(v)) for v in a[e]]
        exact, terms = h0 * g0 + h1 * g1, abs(h0 * g0) + abs(h1 * g1)
        assert abs(Fraction(float(c[e])) - exact) <= abs(exact) / 2 ** 53 + terms * Fraction(65, 64) / 2 ** 56


@pytest.mark.parametrize("h,g", [((1.0, 0.0), (2.0 ** -600, 2.0 ** 600)), ((2.0 ** -100, 0.0), (3.0, 1e300)),
                                 ((0.0, 2.0 ** 90), (1e300, 2.0 ** -700)), ((1.0, 2.0 ** -300), (1.0, 2.0 ** 400)),
                                 ((1.0, 2.0 ** -400), (1.0, 2.0 ** 400)), ((1.0, 5e-324), (1.0, 1.0)),
                                 ((1.25, 0.75), (0.0, 1.0)), ((1.25, 0.75), (0.0, 0.0))])
def test_a_zero_component_does_not_set_the_scale(dot, h, g):
    # exact (or left to FP64) whatever the exponents beside a zero
    c, ok = dot([[*h, *g]])
    exact = Fraction(h[0]) * Fraction(g[0]) + Fraction(h[1]) * Fraction(g[1])
    assert not ok[0] or abs(Fraction(float(c[0])) - exact) <= abs(exact) / 2 ** 52


def thin_cloud(nx, ny, stretch, seed):
    """Jittered nx x ny grid of spacings 1 and 1/stretch, axis-aligned normals, the
    surrounding 3x3 block as neighbours, far-field flags on the border."""
    rng = np.random.default_rng(seed)
    n = nx * ny
    i, j = np.arange(n) % nx, np.arange(n) // nx
    x = i + 0.1 * rng.uniform(-1, 1, n)
    y = (j + 0.1 * rng.uniform(-1, 1, n)) / stretch
    border = (i == 0) | (i == nx - 1) | (j == 0) | (j == ny - 1)
    rows = []
    for p in range(n):
        rows.append([(j[p] + b) * nx + i[p] + a for b in (-1, 0, 1) for a in (-1, 0, 1)
                     if (a or b) and 0 <= i[p] + a < nx and 0 <= j[p] + b < ny])
    off = np.zeros(n + 1, dtype=np.int32)
    off[1:] = np.cumsum([len(r) for r in rows])
    return {"n": n, "x": x, "y": y, "nx": np.zeros(n), "ny": np.ones(n), "flags": np.where(border, 2, 0).astype(np.int32),
            "nbr_offsets": off, "nbr_idx": np.concatenate(rows).astype(np.int32), "wall_order": np.zeros(0, dtype=np.int32)}


def thin_state(cloud, stretch, seed, amp=0.1):
    """A state that varies as fast across the thin direction (per cell) as along the other."""
    rng = np.random.default_rng(seed)
    f = lambda: np.sin(rng.uniform(0.5, 1.0) * cloud["x"] + rng.uniform(0.5, 1.0) * stretch * cloud["y"] + rng.uniform(0, 6))  # noqa: E731
    rho, u, v, p = 1 + amp * f(), 0.5 + amp * f(), amp * f(), (1 + amp * f()) / 1.4
    return np.ascontiguousarray(np.stack([rho, rho * u, rho * v, p / 0.4 + 0.5 * rho * (u * u + v * v)]))


def turned(cloud, U, angle):
    """The cloud with its normals and the state's momentum turned by -angle."""
    c, s = np.cos(angle), np.sin(angle)
    out = dict(cloud)
    out["x"], out["y"] = cloud["x"] * c + cloud["y"] * s, cloud["y"] * c - cloud["x"] * s
    out["nx"], out["ny"] = cloud["nx"] * c + cloud["ny"] * s, cloud["ny"] * c - cloud["nx"] * s
    return out, np.ascontiguousarray(np.stack([U[0], U[1] * c + U[2] * s, U[2] * c - U[1] * s, U[3]]))


def extended_q_derivatives(cloud, U, inner):
    """E13-E15 in numpy's extended precision, and the size of the summands."""
    T = np.longdouble
    U, x, y = U.astype(T), cloud["x"].astype(T), cloud["y"].astype(T)
    n = cloud["n"]
    src, dst = np.repeat(np.arange(n), np.diff(cloud["nbr_offsets"])), cloud["nbr_idx"].astype(np.int64)

    def rows(v):
        return np.stack([np.add.reduceat(c, cloud["nbr_offsets"][:-1]) for c in np.atleast_2d(v)])

    rho, u, v = U[0], U[1] / U[0], U[2] / U[0]
    p = T(2) / T(5) * (U[3] - rho * (u * u + v * v) / 2)
    b = rho / (2 * p)
    q = np.stack([np.log(rho) + T(5) / 2 * np.log(b) - b * (u * u + v * v), 2 * b * u, 2 * b * v, -2 * b])
    dx, dy = x[dst] - x[src], y[dst] - y[src]
    xx, xy, yy = rows(np.stack([dx * dx, dx * dy, dy * dy]))
    det = xx * yy - xy * xy
    ax, ay = (yy[src] * dx - xy[src] * dy) / det[src], (xx[src] * dy - xy[src] * dx) / det[src]
    dq = q[:, dst] - q[:, src]
    gx, gy = rows(ax * dq), rows(ay * dq)
    size = np.abs(q[:, dst]) + np.abs(q[:, src]) + 1     # of a summand, before its weight
    for _ in range(inner):
        cx, cy = dx * (gx[:, dst] - gx[:, src]) / 2, dy * (gy[:, dst] - gy[:, src]) / 2
        size = size + (np.abs(dx) * (np.abs(gx[:, dst]) + np.abs(gx[:, src])) + np.abs(dy) * (np.abs(gy[:, dst]) + np.abs(gy[:, src]))) / 2
        gx, gy = rows(ax * (dq - cx - cy)), rows(ay * (dq - cx - cy))
    return (gx, gy), (rows(np.abs(ax) * size), rows(np.abs(ay) * size))


@pytest.mark.gpu
@pytest.mark.parametrize("stretch", [1.0, 2.0 ** 10, 2.0 ** 20, 2.0 ** 30])
def test_q_derivatives_of_a_stretched_cloud(stretch):
    """Per point the sum of up to 8 weighted differences over K + 1 = 3 passes. A
    weight of the closed 2 x 2 solve carries at most 12 roundings (offsets, sums of
    products, determinant and quotient; the determinant of these jittered blocks
    keeps above 0.9 of xx yy), q 4, an inner pass 8 per summand more: 64 units of
    2^-53 of the summands' size, whatever the stretching."""
    import torch

    from paper_2403_13287_gb300.lskum import Solver
    c = thin_cloud(41, 37, stretch, seed=3)
    U = thin_state(c, stretch, seed=5)
    s = Solver(c, order=2, inner_iters=2, mach=0.5, aoa_deg=0.0)
    got = [t.cpu().numpy() for t in s.q_derivatives(torch.from_numpy(U).cuda())]
    s.close()
    want, size = extended_q_derivatives(c, U, 2)
    for g, w, z in zip(got, want, size):
        err = np.abs(g - w) / z
        assert np.all(err <= 64 * 2.0 ** -53), float(err.max() * 2.0 ** 53)


@pytest.mark.gpu
@pytest.mark.parametrize("limiter", [0.0, 1.0])
def test_products_of_a_stretched_cloud(limiter):
    """Sampled entries of U_bar and y_bar at 1000 : 1 against complex-step
    derivatives, at the VJP tests' 1e-10 of the largest."""
    import torch

    import oracle
    from oracle import lskum_jvp
    from paper_2403_13287_gb300.lskum import Solver
    c = thin_cloud(31, 29, 1000.0, seed=4)
    n = c["n"]
    U = thin_state(c, 1000.0, seed=6)
    rng = np.random.default_rng(1)
    Rb = rng.standard_normal((4, n))
    s = Solver(c, order=2, inner_iters=2, mach=0.5, aoa_deg=0.0, limiter_K=limiter)
    Ub, xb, yb = (t.cpu().numpy() for t in s.residual_vjp(torch.from_numpy(Rb).cuda(), torch.from_numpy(U).cuda()))
    s.close()
    ent = [("U", int(rng.integers(4)), int(k)) for k in rng.choice(n, 40, replace=False)]
    ent += [("y", int(k)) for k in rng.choice(n, 20, replace=False)]
    want = lskum_jvp.vjp_entries(c, oracle.split_stencils(c), U, Rb, ent, order=2, inner=2, limiter=limiter)
    got = np.array([Ub[e[1], e[2]] if e[0] == "U" else yb[e[1]] for e in ent])
    for kind in "Uy":
        k = [i for i, e in enumerate(ent) if e[0] == kind]
        assert np.all(np.abs(got - want)[k] <= 1e-10 * np.abs(want[k]).max())


@pytest.mark.gpu
def test_products_of_a_stretched_cloud_across_both_axes():
    """Stretched A = 4096 : 1 at half a radian to the axes. The determinants of the
    closed 2 x 2 solves cancel to A^-2 of their products, so weights, and sums of
    them, carry a few units of 2^-53 A^2 on either side: 16 of them of the largest
    entry."""
    import torch

    import oracle
    from oracle import lskum_jvp
    from paper_2403_13287_gb300.lskum import Solver
    A = 4096.0
    c = thin_cloud(31, 29, A, seed=3)
    c, U = turned(c, thin_state(c, A, seed=5), 0.5)
    n = c["n"]
    rng = np.random.default_rng(2)
    Rb = rng.standard_normal((4, n))
    s = Solver(c, order=2, inner_iters=2, mach=0.5, aoa_deg=0.0)
    Ub, xb, yb = (t.cpu().numpy() for t in s.residual_vjp(torch.from_numpy(Rb).cuda(), torch.from_numpy(U).cuda()))
    s.close()
    ent = [("U", int(rng.integers(4)), int(k)) for k in rng.choice(n, 20, replace=False)]
    ent += [(d, int(k)) for d in "xy" for k in rng.choice(n, 30, replace=False)]
    want = lskum_jvp.vjp_entries(c, oracle.split_stencils(c), U, Rb, ent, order=2, inner=2)
    got = np.array([Ub[e[1], e[2]] if e[0] == "U" else (xb if e[0] == "x" else yb)[e[1]] for e in ent])
    for kind in "Uxy":
        k = [i for i, e in enumerate(ent) if e[0] == kind]
        assert np.all(np.abs(got - want)[k] <= 16 * A * A * 2.0 ** -53 * np.abs(want[k]).max()), kind


@pytest.mark.gpu
@pytest.mark.parametrize("axis", [0, 1])
def test_slow_gas_in_thin_stencils(axis):
    """Velocities of 1e-8 in a cloud stretched 2^30 : 1, either way: the momentum
    across the weak direction is carried by the transverse fluxes, rho u_t u_n P
    with a small u, times the strong direction's weights. First-order residual at
    1e-12 of each component's largest entry (the parity tests' bar), and its product
    with a cotangent of that component, at the VJP tests' 1e-10."""
    import torch

    import oracle
    from oracle import lskum_jvp
    from paper_2403_13287_gb300.lskum import Solver
    A = 2.0 ** 30 if axis == 0 else 2.0 ** -30
    c = thin_cloud(23, 21, A, seed=3)
    n = c["n"]
    U = thin_state(c, A, seed=5)
    u = U[1:3] / U[0]
    U[3] += 0.5 * U[0] * ((1e-16 - 1) * (u * u).sum(0))
    U[1:3] *= 1e-8
    s = Solver(c, order=1, inner_iters=0, mach=0.5, aoa_deg=0.0)
    R = s.residual(torch.from_numpy(U).cuda()).cpu().numpy()
    m = oracle.split_stencils(c)
    Ro = oracle.residual(c, m, U, order=1, inner=0)
    k = 1 + axis
    for j in range(4):
        assert np.abs(R[j] - Ro[j]).max() <= 1e-12 * np.abs(Ro[j]).max(), j
    rng = np.random.default_rng(1)
    Rb = np.zeros((4, n))
    Rb[k] = rng.standard_normal(n)
    Ub, xb, yb = (t.cpu().numpy() for t in s.residual_vjp(torch.from_numpy(Rb).cuda(), torch.from_numpy(U).cuda()))
    s.close()
    ent = [("U", int(rng.integers(4)), int(e)) for e in rng.choice(n, 20, replace=False)]
    ent += [("y" if axis == 0 else "x", int(e)) for e in rng.choice(n, 20, replace=False)]
    want = lskum_jvp.vjp_entries(c, m, U, Rb, ent, order=1, inner=0)
    got = np.array([Ub[e[1], e[2]] if e[0] == "U" else (xb if e[0] == "x" else yb)[e[1]] for e in ent])
    for kind in "Uxy":
        i = [j for j, e in enumerate(ent) if e[0] == kind]
        if i:
            assert np.all(np.abs(got - want)[i] <= 1e-10 * np.abs(want[i]).max()), kind
