"""The work that users of q-LSKUM on the GPU have it do, as timed cases.

A case names a synthetic NACA 0012 cloud (W wall points, L layers: W (L + 1)
points), the scheme and the call. Kinds of call:

- march:    a solve from a given state: set_state, `iters` pseudo-time
            iterations, the new state (and the forces where a design loop
            reads them); returns the residue history and the state.
- batch:    the same for several clouds under several free streams in one
            context (Solver.batch).
- residual: R(U) of one state (lskum_residual).
- vjp:      residual and its reverse pass through torch autograd
            (residual_fn): R, and the gradients of <R, R_bar> in U and in the
            coordinates.
- vjp32:    the FP32 product of a mixed context (residual_vjp(fp32=True)), in
            U only, as its documentation advises.
- step_vjp: one pseudo-time iteration in reverse (the unit of an unrolled
            adjoint sweep): cotangents of U and of the coordinates.

exact() restates the scheme in plain FP64 torch, vectorised over the stencil
edges, with derivatives by torch autograd.
"""
import math

import numpy as np
import torch

from paper_2403_13287_gb300.cloudgen import naca0012_cloud, smooth_state
from paper_2403_13287_gb300.lskum import Solver, residual_fn

GAMMA = 1.4
CFL = 0.2

_BASE = {"kind": "march", "W": 0, "L": 0, "order": 2, "inner": 3, "rk4": True, "mach": 1.2, "aoa": 0.0, "limiter": 0.0,
         "mixed": False, "kinetic": False, "reorder": 1, "shuffle": True, "iters": 1, "forces": False, "tuned": False,
         "clouds": 1, "streams": 1}


def _case(name=None, **kw):
    c = dict(_BASE, **kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call: one residual of a coarse cloud in the caller's order, as a residual check or an outer
        # Newton / time integrator of the user's own makes it, thousands of times over
        _case("residual_fp64_3k", kind="residual", W=130, L=24, mach=0.63, aoa=2.0, reorder=0, shuffle=False),
        # a coarse first-order solve with its forces: the start-up phase and the angle-of-attack sweeps
        _case("march_fp64_first_order_10k", W=320, L=30, order=1, inner=0, rk4=False, mach=0.63, aoa=2.0, iters=20,
              forces=True),
        # the transonic workload: second order, limited, RK4, on a medium cloud
        _case("march_fp64_rk4_limited_160k", W=512, L=311, mach=0.85, aoa=1.0, limiter=1.0, iters=2),
        # the published benchmark's own condition: forward Euler, unlimited, Mach 0.63
        _case("march_fp64_euler_640k", W=1024, L=624, rk4=False, mach=0.63, aoa=2.0, iters=2),
        # the headline workload: 2.5 million points, RK4, Mach 1.2, limited, in FP64 ...
        _case("march_fp64_rk4_limited_2p5m", W=2560, L=975, limiter=1.0),
        # ... and in the mixed form, launch shapes tuned once as the documentation tells a long run to do
        _case("march_mixed_rk4_limited_2p5m", W=2560, L=975, limiter=1.0, mixed=True, iters=5, tuned=True),
        # the transonic workload in the mixed form with the default launch shapes, as a short run uses it
        _case("march_mixed_rk4_limited_160k", W=512, L=311, mach=0.85, aoa=1.0, limiter=1.0, mixed=True, iters=10),
        # a small design study: uneven clouds under three free streams each, advanced together
        _case("batch_mixed_12", kind="batch", W=384, L=233, mach=0.5, limiter=1.0, mixed=True, clouds=4, streams=3,
              iters=2),
        # kinetic wall and far-field conditions, reverse Cuthill-McKee numbering
        _case("march_mixed_kinetic_93k", W=402, L=231, mach=0.85, aoa=1.0, limiter=1.0, mixed=True, kinetic=True,
              reorder=2, iters=4),
        # gradient of a residual functional in the state and in the shape (autograd, FP64)
        _case("vjp_fp64_93k", kind="vjp", W=402, L=231, mach=0.63, aoa=2.0),
        # transposed product of an adjoint solver's inner iteration, in FP32, at the adjoint workload's size
        _case("vjp_fp32_640k", kind="vjp32", W=1024, L=624, mach=0.63, aoa=2.0, mixed=True),
        # one limited RK4 iteration in reverse: the unit of an unrolled sensitivity sweep
        _case("step_vjp_fp64_40k", kind="step_vjp", W=256, L=155, limiter=1.0),
    ]


def _cloud_size(rng, lo, hi):
    """W (even) and L of a cloud of lo..hi points, log-uniform; near-isotropic layering, as in the named clouds."""
    n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    ratio = rng.uniform(0.40, 0.60)
    W = 2 * max(40, round(math.sqrt(n / ratio) / 2))
    return W, max(24, round(n / W) - 1)


def draw(rng):
    kind = rng.choice(["march", "march", "march", "march", "residual", "batch", "vjp", "vjp32", "step_vjp"])
    mach, aoa = rng.choice([(0.63, 2.0), (0.85, 1.0), (1.2, 0.0)])
    limiter = 0.0 if mach < 0.7 else 1.0
    reorder = rng.choice([0, 1, 1, 2])
    c = _case(kind=kind, mach=mach, aoa=aoa, limiter=limiter, reorder=reorder, shuffle=reorder != 0)
    if kind == "march":
        c["mixed"] = rng.random() < 0.5
        c["rk4"] = rng.random() < 0.6
        c["kinetic"] = rng.random() < 0.25
        c["forces"] = rng.random() < 0.25
        if rng.random() < 0.2:
            c.update(order=1, inner=0, limiter=0.0)
        c["W"], c["L"] = _cloud_size(rng, 3e3, 1e6 if c["mixed"] else 6.5e5)
        c["iters"] = rng.randint(1, 3)
    elif kind == "residual":
        c["mixed"] = rng.random() < 0.5
        c["W"], c["L"] = _cloud_size(rng, 3e3, 3e5)
    elif kind == "batch":
        c.update(reorder=1, shuffle=True, mixed=True, mach=0.5, limiter=1.0, clouds=rng.randint(2, 4), streams=rng.randint(1, 3),
                 iters=rng.randint(1, 3))
        c["W"], c["L"] = _cloud_size(rng, 2e4, 1e5)
    elif kind == "vjp32":
        c.update(mixed=True, limiter=0.0)
        c["W"], c["L"] = _cloud_size(rng, 1e4, 6e5)
    else:
        c["W"], c["L"] = _cloud_size(rng, 5e3, 1.5e5 if kind == "vjp" else 8e4)
    return c


# --------------------------------------------------------------------------- inputs

def _cloud(case, seed, k=0):
    """Cloud k of a case: its jitter and point order come from the seed; a batch's clouds shrink with k."""
    W, L = case["W"], case["L"]
    if k:
        W, L = 2 * round(W * 0.8 ** k / 2), round(L * 0.8 ** k)
    return naca0012_cloud(W, L, seed=1000 + 10 * (seed % 100003) + k, shuffle=case["shuffle"])


def _streams(case):
    """(Mach, angle of attack) of a batch's free streams."""
    return [(case["mach"] + 0.3 * j, -1.0 + 2.0 * j) for j in range(case["streams"])]


def _inputs(case, seed):
    """The clouds, free streams and states of a case: lists of (cloud, mach, aoa, U)."""
    out = []
    for k in range(case["clouds"]):
        cloud = _cloud(case, seed, k)
        for j, (m, a) in enumerate(_streams(case) if case["kind"] == "batch" else [(case["mach"], case["aoa"])]):
            out.append((cloud, m, a, smooth_state(cloud, m, a, amp=0.05, seed=seed + 17 * k + j)))
    return out


def _cotangent(cloud, seed):
    """A cotangent of unit size (of R, or of the next state), zero mean, one independent value per point."""
    return np.random.Generator(np.random.PCG64(seed + 5)).standard_normal((4, cloud["n"]))


def prepare(case, seed):
    ins = _inputs(case, seed)
    cloud, mach, aoa, _ = ins[0]
    kw = dict(order=case["order"], inner_iters=case["inner"], time_scheme=1 if case["rk4"] else 0, cfl=CFL,
              limiter_K=case["limiter"], precision=1 if case["mixed"] else 0, reorder=case["reorder"],
              boundary=1 if case["kinetic"] else 0)
    if case["kind"] == "batch":
        solver = Solver.batch([i[:3] for i in ins], **kw)
    else:
        solver = Solver(cloud, mach=mach, aoa_deg=aoa, **kw)
    U = torch.from_numpy(np.ascontiguousarray(np.concatenate([i[3] for i in ins], axis=1))).cuda()
    s = {"case": case, "solver": solver, "U": U, "out": torch.empty_like(U)}
    if case["tuned"]:
        solver.set_state(U)
        solver.autotune()
    if case["kind"] in ("vjp", "vjp32", "step_vjp"):
        s["bar"] = torch.from_numpy(_cotangent(cloud, seed)).cuda()
        s["xy"] = torch.from_numpy(np.stack([cloud["x"], cloud["y"]])).cuda()
    return s


def run(state):
    case, solver, U = state["case"], state["solver"], state["U"]
    kind = case["kind"]
    if kind in ("march", "batch"):
        solver.set_state(U)
        history = solver.step(case["iters"])
        got = {"history": history, "U": solver.get_state(out=state["out"])}
        if case["forces"]:
            cl, cd, cp = solver.forces()
            got["forces"] = np.array([cl, cd])
            got["cp"] = cp
        return got
    if kind == "residual":
        return {"R": solver.residual(U, out=state["out"])}
    if kind == "vjp":
        u = U.detach().requires_grad_()
        xy = state["xy"].detach().requires_grad_()
        R = residual_fn(solver, u, xy)
        R.backward(state["bar"])
        return {"R": R.detach(), "U_bar": u.grad, "xy_bar": xy.grad}
    if kind == "vjp32":
        return {"U_bar": solver.residual_vjp(state["bar"], U, want_xy=False, fp32=True)[0]}
    Ub, xb, yb = solver.step_vjp(state["bar"], U=U)
    return {"U_bar": Ub, "x_bar": xb, "y_bar": yb}


# Mean number of neighbours of these clouds, and FP operations per edge (a fused multiply-add counts two) of one
# first-order solve of the q-derivatives, one inner iteration, the limiter and the split fluxes of both states.
_DEGREE = 8.14
_FLOPS = {"first": 20, "inner": 32, "limiter": 16, "flux": 285}


def work(case):
    """Bytes: U (and a cotangent) in, the results out, the cloud (coordinates, normals, flags, neighbour lists) once.
    Flops: the edges' arithmetic of every residual of the pass; a reverse pass counts twice its forward."""
    n = sum((2 * round(case["W"] * 0.8 ** k / 2)) * (round(case["L"] * 0.8 ** k) + 1) for k in range(case["clouds"]))
    copies = case["streams"] if case["kind"] == "batch" else 1
    cloud = n * (16 + 16 + 1 + 4 + 4 * _DEGREE)
    residual = _FLOPS["flux"]
    if case["order"] == 2:
        residual += _FLOPS["first"] + case["inner"] * _FLOPS["inner"] + (_FLOPS["limiter"] if case["limiter"] else 0)
    stages = 4 if case["rk4"] else 1
    per = {"march": case["iters"] * stages, "batch": case["iters"] * stages, "residual": 1, "vjp": 3, "vjp32": 3,
           "step_vjp": 3 * stages}[case["kind"]]
    vectors = {"march": 2, "batch": 2, "residual": 2, "vjp": 4.5, "vjp32": 3, "step_vjp": 3.5}[case["kind"]]
    return {"bytes": cloud + copies * n * 32 * vectors, "flops": copies * n * _DEGREE * residual * per}


# --------------------------------------------------------------------------- the scheme in plain FP64 torch

def _freestream(mach, aoa, dev):
    a = math.radians(aoa)
    u, v, p = mach * math.cos(a), mach * math.sin(a), 1.0 / GAMMA
    return torch.tensor([1.0, u, v, p / (GAMMA - 1.0) + 0.5 * (u * u + v * v)], dtype=torch.float64, device=dev)


def _q_of(U):
    rho, u, v = U[0], U[1] / U[0], U[2] / U[0]
    p = (GAMMA - 1.0) * (U[3] - 0.5 * rho * (u * u + v * v))
    b = 0.5 * rho / p
    return torch.stack([torch.log(rho) + torch.log(b) / (GAMMA - 1.0) - b * (u * u + v * v), 2 * b * u, 2 * b * v, -2 * b])


def _split_flux(q, tx, ty, sign, along):
    """The kinetic split flux of q along t (along=True) or n, sign +1 or -1 per edge; frame order [mass, s, n, energy]."""
    b = -0.5 * q[3]
    u, v = q[1] / (2 * b), q[2] / (2 * b)
    rho = torch.exp(q[0] + b * (u * u + v * v) - torch.log(b) / (GAMMA - 1.0))
    p = rho / (2 * b)
    us, un = u * tx + v * ty, -u * ty + v * tx        # n = (-ty, tx)
    d, t = (us, un) if along else (un, us)
    S = d * torch.sqrt(b)
    A = 0.5 * (1.0 + sign * torch.erf(S))
    B = sign * torch.exp(-S * S) / (2.0 * torch.sqrt(math.pi * b))
    E = p / (GAMMA - 1.0) + 0.5 * rho * (u * u + v * v)
    m = rho * (d * A + B)
    g1 = (p + rho * d * d) * A + rho * d * B
    g3 = (E + p) * d * A + (E + 0.5 * p) * B
    return torch.stack([m, g1, t * m, g3] if along else [m, t * m, g1, g3])


class _Scheme:
    """The residual and the pseudo-time step of one cloud, differentiable in U, x and y."""

    def __init__(self, cloud, mach, aoa, case):
        self.dev = dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        t = lambda a: torch.as_tensor(np.ascontiguousarray(a)).to(dev)  # noqa: E731
        self.case, self.n = case, cloud["n"]
        self.x, self.y, self.nx, self.ny = (t(cloud[k]) for k in ("x", "y", "nx", "ny"))
        self.flag = t(cloud["flags"]).long()
        self.row = torch.repeat_interleave(torch.arange(self.n, device=dev), t(np.diff(cloud["nbr_offsets"])).long())
        self.idx = t(cloud["nbr_idx"]).long()
        self.wall_order = t(cloud["wall_order"]).long()
        self.mach, self.aoa = mach, aoa
        self.Uinf = _freestream(mach, aoa, dev)
        self.geometry(self.x, self.y)

    def sum(self, v, row):
        return torch.zeros((v.shape[0], self.n), dtype=torch.float64, device=self.dev).index_add(1, row, v)

    def first(self, v, row, largest):
        """Per row, the first entry (in row order) with the largest (smallest) value."""
        v = v.detach()
        far = -math.inf if largest else math.inf
        m = torch.full((self.n,), far, dtype=torch.float64, device=self.dev)
        m = m.scatter_reduce(0, row, v, "amax" if largest else "amin")
        e = torch.arange(row.numel(), device=self.dev)
        none = row.numel()
        at = torch.full((self.n,), none, dtype=torch.long, device=self.dev)
        return at.scatter_reduce(0, row, torch.where(v == m[row], e, torch.full_like(e, none)), "amin")

    def geometry(self, x, y):
        """Offsets, least-squares weights (full and sub-stencil), nearest distances; images in the kinetic mode."""
        row, idx = self.row, self.idx
        dx, dy = x[idx] - x[row], y[idx] - y[row]
        nx, ny = self.nx[row], self.ny[row]
        ds, dn = dx * ny - dy * nx, dx * nx + dy * ny
        near = self.first(dx * dx + dy * dy, row, largest=False)
        self.dmin = torch.sqrt((dx * dx + dy * dy)[near])
        self.erow, self.eidx, self.image = row, idx, None
        if self.case["kinetic"]:
            # wall and far-field points also see the mirror images of their neighbours off the tangent line
            k = torch.nonzero((self.flag[row] != 0) & (dn != 0)).squeeze(1)
            self.erow, self.eidx = torch.cat([row, row[k]]), torch.cat([idx, idx[k]])
            self.image = torch.cat([torch.zeros_like(row), self.flag[row[k]]])       # 1 wall, 2 far field
            dx = torch.cat([dx, dx[k] - 2 * dn[k] * nx[k]])
            dy = torch.cat([dy, dy[k] - 2 * dn[k] * ny[k]])
            ds, dn = torch.cat([ds, ds[k]]), torch.cat([dn, -dn[k]])
        row = self.erow
        self.dx, self.dy = dx, dy
        xx, xy, yy = self.sum(torch.stack([dx * dx, dx * dy, dy * dy]), row)
        det = xx * yy - xy * xy
        self.a = torch.stack([(yy[row] * dx - xy[row] * dy) / det[row], (xx[row] * dy - xy[row] * dx) / det[row]])
        self.sgn, self.w = [], []
        f = self.flag[row]
        for along, d in ((True, ds), (False, dn)):
            w = torch.zeros_like(d)
            for positive in (True, False):                 # G+ takes the members behind, G- those ahead
                member = d < 0 if positive else d > 0
                if not self.case["kinetic"]:
                    member = member & (f != 2) & ((f != 1) | along | (not positive))
                k = torch.nonzero(member).squeeze(1)
                s, m, r = ds[k], dn[k], row[k]
                ss, sn, nn = self.sum(torch.stack([s * s, s * m, m * m]), r)
                D = (ss * nn - sn * sn)[r]
                wk = (nn[r] * s - sn[r] * m) / D if along else (ss[r] * m - sn[r] * s) / D
                w = w.index_add(0, k, wk)
            self.w.append(w)
            self.sgn.append(torch.where(d.detach() < 0, 1.0, -1.0).to(torch.float64))

    def reflect(self, a, b):
        nx, ny = self.nx[self.erow], self.ny[self.erow]
        c = a * nx + b * ny
        return a - 2 * c * nx, b - 2 * c * ny

    def far(self, v):
        """A member's values v ([4, edges], of the neighbour) as its image carries them (value part)."""
        if self.image is None:
            return v
        ra, rb = self.reflect(v[1], v[2])
        w = self.image == 1
        return torch.stack([v[0], torch.where(w, ra, v[1]), torch.where(w, rb, v[2]), v[3]])

    def shift(self, gx, gy):
        """d . grad q of every member, the gradient being the neighbour's (reflected, or none, for an image)."""
        dx, dy = self.dx, self.dy
        if self.image is not None:
            rx, ry = self.reflect(dx, dy)
            w = self.image == 1
            dx, dy = torch.where(w, rx, dx), torch.where(w, ry, dy)
        c = dx * gx[:, self.eidx] + dy * gy[:, self.eidx]
        if self.image is not None:
            c = torch.where(self.image == 2, torch.zeros_like(c), self.far(c))
        return c

    def member_q(self, q):
        v = self.far(q[:, self.eidx])
        if self.image is not None:
            v = torch.where(self.image == 2, _q_of(self.Uinf)[:, None], v)
        return v

    def gradients(self, q):
        row, dx, dy = self.erow, self.dx, self.dy
        dq = self.member_q(q) - q[:, row]
        gx, gy = self.sum(self.a[0] * dq, row), self.sum(self.a[1] * dq, row)
        for _ in range(self.case["inner"]):
            c = dq - 0.5 * (self.shift(gx, gy) - (dx * gx[:, row] + dy * gy[:, row]))
            gx, gy = self.sum(self.a[0] * c, row), self.sum(self.a[1] * c, row)
        K = self.case["limiter"]
        if K:
            # Venkatakrishnan: phi = f(x, d) where x < 2 d, else 1; x = min(D+, -D-), d the largest |shift|
            eps = (K * self.dmin) ** 3
            phi = []
            z = torch.zeros(self.n, dtype=torch.float64, device=self.dev)
            for k in range(4):
                hi, lo = dq[k][self.first(dq[k], row, True)], dq[k][self.first(dq[k], row, False)]
                hi, lo = torch.where(hi > 0, hi, z), torch.where(lo < 0, lo, z)
                c = 0.5 * (dx * gx[k][row] + dy * gy[k][row])
                d = c.abs()[self.first(c.abs(), row, True)]
                X = torch.where(hi <= -lo, hi, -lo)
                f = (X * X + eps + 2 * X * d) / (X * X + 2 * d * d + X * d + eps)
                phi.append(torch.where(X < 2 * d, f, torch.ones_like(f)))
            phi = torch.stack(phi)
            gx, gy = phi * gx, phi * gy
        return gx, gy

    def residual(self, U):
        q = _q_of(U)
        row, dx, dy = self.erow, self.dx, self.dy
        qi, q0 = self.member_q(q), q[:, row]
        if self.case["order"] == 2:
            gx, gy = self.gradients(q)
            far = None if self.image is None else self.image == 2
            # (the reconstruction of a far-field image is the free stream: its shift is zero)
            qi = qi - 0.5 * self.shift(gx, gy) if far is None else torch.where(far, qi, qi - 0.5 * self.shift(gx, gy))
            q0 = q0 - 0.5 * (dx * gx[:, row] + dy * gy[:, row])
        tx, ty = self.ny[row], -self.nx[row]
        R = 0
        for along, w, sgn in ((True, self.w[0], self.sgn[0]), (False, self.w[1], self.sgn[1])):
            dG = _split_flux(qi, tx, ty, sgn, along) - _split_flux(q0, tx, ty, sgn, along)
            R = R + self.sum(w * dG, row)
        return torch.stack([R[0], R[1] * self.ny + R[2] * self.nx, -R[1] * self.nx + R[2] * self.ny, R[3]])

    def boundary(self, U):
        wall, mn = self.flag == 1, U[1] * self.nx + U[2] * self.ny
        U = torch.stack([U[0], torch.where(wall, U[1] - mn * self.nx, U[1]), torch.where(wall, U[2] - mn * self.ny, U[2]),
                         U[3]])
        return U if self.case["kinetic"] else torch.where(self.flag == 2, self.Uinf[:, None], U)

    def step(self, U):
        rho, u, v = U[0], U[1] / U[0], U[2] / U[0]
        p = (GAMMA - 1.0) * (U[3] - 0.5 * rho * (u * u + v * v))
        dt = CFL * self.dmin / (torch.sqrt(u * u + v * v) + 3.0 * torch.sqrt(p / rho))
        R0 = self.residual(U)
        if not self.case["rk4"]:
            return self.boundary(U - dt * R0), R0
        R1 = self.residual(self.boundary(U - 0.5 * dt * R0))
        R2 = self.residual(self.boundary(U - 0.5 * dt * R1))
        R3 = self.residual(self.boundary(U - dt * R2))
        return self.boundary(U - dt / 6.0 * (R0 + 2 * R1 + 2 * R2 + R3)), R0

    def forces(self, U):
        o = self.wall_order
        rho, u, v = U[0, o], U[1, o] / U[0, o], U[2, o] / U[0, o]
        p = (GAMMA - 1.0) * (U[3, o] - 0.5 * rho * (u * u + v * v))
        cp = (p - 1.0 / GAMMA) / (0.5 * self.mach ** 2)
        x, y = self.x[o], self.y[o]
        seg = torch.hypot(torch.roll(x, -1) - x, torch.roll(y, -1) - y)
        ds = 0.5 * (seg + torch.roll(seg, 1))
        fx, fy, a = -(cp * self.nx[o] * ds).sum(), -(cp * self.ny[o] * ds).sum(), math.radians(self.aoa)
        return torch.stack([fy * math.cos(a) - fx * math.sin(a), fx * math.cos(a) + fy * math.sin(a)]), cp


def exact(case, seed):
    ins = _inputs(case, seed)
    if case["kind"] in ("march", "batch", "residual"):
        with torch.no_grad():
            histories, states, more = [], [], {}
            for cloud, mach, aoa, U in ins:
                s = _Scheme(cloud, mach, aoa, case)
                U = torch.from_numpy(U).to(s.dev)
                if case["kind"] == "residual":
                    return {"R": s.residual(U)}
                h = []
                for _ in range(case["iters"]):
                    U, R = s.step(U)
                    h.append(R[0].square().sum().sqrt() / s.n)
                histories.append(torch.stack(h))
                states.append(U)
                if case["forces"]:
                    more["forces"], more["cp"] = s.forces(U)
            history = torch.stack(histories, dim=1) if len(ins) > 1 else histories[0]
            return {"history": history, "U": torch.cat(states, dim=1), **more}
    cloud, mach, aoa, U = ins[0]
    s = _Scheme(cloud, mach, aoa, case)
    U = torch.from_numpy(U).to(s.dev).requires_grad_()
    bar = torch.from_numpy(_cotangent(cloud, seed)).to(s.dev)
    if case["kind"] == "vjp32":
        return {"U_bar": torch.autograd.grad((s.residual(U) * bar).sum(), U)[0]}
    x, y = s.x.clone().requires_grad_(), s.y.clone().requires_grad_()
    s.geometry(x, y)
    out = s.residual(U) if case["kind"] == "vjp" else s.step(U)[0]
    Ub, xb, yb = torch.autograd.grad((out * bar).sum(), (U, x, y))
    if case["kind"] == "vjp":
        return {"R": out.detach(), "U_bar": Ub, "xy_bar": torch.stack([xb, yb])}
    return {"U_bar": Ub, "x_bar": xb, "y_bar": yb}
