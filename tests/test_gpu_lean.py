"""Contexts without the arrays that only save time (lskum_set_lean): the same bits,
and the memory is given back (needs a GPU)."""
import numpy as np
import pytest

from paper_2403_13287_gb300.cloudgen import naca0012_cloud, smooth_state

pytestmark = pytest.mark.gpu


def _everything(s, U):
    import torch
    out = {"R": s.residual(U)}
    out["qx"], out["qy"] = s.q_derivatives(U)
    s.set_state(U)
    out["history"] = torch.from_numpy(s.step(3))
    out["state"] = torch.from_numpy(s.get_state())
    return {k: v.cpu().numpy() for k, v in out.items()}


@pytest.mark.parametrize("order,limiter,boundary,time_scheme", [(2, 0.0, 0, 1), (2, 1.0, 0, 0), (2, 1.0, 1, 1), (1, 0.0, 0, 1)])
def test_forward_is_the_same_without_optional_arrays(order, limiter, boundary, time_scheme):
    """Before, lean, and back again on one context, the step graphs replayed in
    between."""
    import torch

    from paper_2403_13287_gb300.lskum import Solver
    c = naca0012_cloud(180, 99, seed=3, shuffle=True)
    U = torch.from_numpy(smooth_state(c, 0.85, 1.0, amp=0.05, seed=9)).cuda()
    s = Solver(c, order=order, inner_iters=3 if order == 2 else 0, time_scheme=time_scheme, limiter_K=limiter, mach=0.85,
               aoa_deg=1.0, reorder=1, boundary=boundary)
    got = []
    for lean in (None, True, False):
        if lean is not None:
            s.set_lean(lean)
        got.append(_everything(s, U))
    s.close()
    for other in got[1:]:
        for k in got[0]:
            assert np.array_equal(got[0][k], other[k]), k


def test_memory_is_given_back():
    """16 B per edge of an FP64 context (21 MB here; the device hands out pieces of
    2 MB), none of a mixed one."""
    import torch

    from paper_2403_13287_gb300.lskum import Solver
    c = naca0012_cloud(512, 311, seed=3)
    for precision, want in ((0, 16 * c["nbr_idx"].size), (1, 0)):
        s = Solver(c, order=2, inner_iters=3, mach=0.85, aoa_deg=1.0, precision=precision, reorder=1)
        free0 = torch.cuda.mem_get_info()[0]
        s.set_lean()
        free1 = torch.cuda.mem_get_info()[0]
        s.set_lean(False)
        free2 = torch.cuda.mem_get_info()[0]
        s.close()
        assert abs((free1 - free0) - want) <= 4 << 20 and free2 == free0


def test_lean_takes_0_or_1():
    from paper_2403_13287_gb300.lskum import LSKUM_ERR_ARG, Solver
    s = Solver(naca0012_cloud(34, 12, seed=1), order=2, mach=0.5, aoa_deg=0.0)
    assert s._L.lskum_set_lean(s._ctx, 2) == LSKUM_ERR_ARG and s._L.lskum_set_lean(s._ctx, -1) == LSKUM_ERR_ARG
    assert s._L.lskum_set_lean(None, 1) == LSKUM_ERR_ARG
    s.close()


@pytest.mark.parametrize("precision,fp32,limiter,order,gamma", [(0, False, 1.0, 2, 1.4), (0, False, 0.0, 1, 1.4),
                                                                (0, False, 0.0, 2, 1.3), (1, True, 0.0, 2, 1.4), (1, False, 0.0, 2, 1.4)])
def test_products_are_the_same_without_optional_arrays(precision, fp32, limiter, order, gamma):
    """Residual product (FP64 of both contexts, FP32), U alone and with coordinates:
    with the arrays, without, and with them again on one context."""
    import torch

    from paper_2403_13287_gb300.lskum import Solver
    c = naca0012_cloud(180, 99, seed=3, shuffle=True)
    U = torch.from_numpy(smooth_state(c, 0.85, 1.0, amp=0.05, seed=9, gamma=gamma)).cuda()
    Rb = torch.from_numpy(np.random.default_rng(1).standard_normal((4, c["n"]))).cuda()
    s = Solver(c, order=order, inner_iters=3 if order == 2 else 0, limiter_K=limiter, mach=0.85, aoa_deg=1.0, gamma=gamma,
               reorder=1, precision=precision)
    got = []
    for lean in (None, True, False):
        if lean is not None:
            s.set_lean(lean)
        for _ in range(2):
            out = s.residual_vjp(Rb, U, fp32=fp32)
            got.append([t.cpu().numpy() for t in out] + [s.residual_vjp(Rb, U, want_xy=False, fp32=fp32)[0].cpu().numpy()])
            s.residual(U)
    s.close()
    for other in got[1:]:
        for p, q in zip(got[0], other):
            assert np.array_equal(p, q)


@pytest.mark.parametrize("limiter,order,time_scheme,want_xy", [(0.0, 2, 1, True), (1.0, 2, 1, True), (1.0, 2, 1, False),
                                                               (0.0, 1, 1, True), (1.0, 2, 0, True)])
def test_step_products_are_the_same_without_optional_arrays(limiter, order, time_scheme, want_xy):
    """With every RK stage's forward kept, and with each run again in the reverse
    sweep: the same bits, first product and repeated ones, another state in between."""
    import torch

    from paper_2403_13287_gb300.lskum import Solver
    c = naca0012_cloud(130, 24, seed=11, shuffle=True)
    U = [torch.from_numpy(smooth_state(c, 0.85, 1.0, amp=0.05, seed=k)).cuda() for k in (9, 10)]
    bar = torch.from_numpy(np.random.default_rng(1).standard_normal((4, c["n"]))).cuda()
    kw = dict(order=order, inner_iters=3 if order == 2 else 0, time_scheme=time_scheme, limiter_K=limiter, mach=0.85,
              aoa_deg=1.0, reorder=1)
    got = []
    kept, lean = Solver(c, **kw), Solver(c, **kw)
    lean.set_lean()
    for s in (kept, lean):
        got.append([t.cpu().numpy() for u in (U[0], U[1], U[0]) for t in s.step_vjp(bar, U=u, want_xy=want_xy) if t is not None])
    kept.set_lean()
    got.append([t.cpu().numpy() for u in (U[0], U[1], U[0]) for t in kept.step_vjp(bar, U=u, want_xy=want_xy) if t is not None])
    kept.close()
    lean.close()
    for other in got[1:]:
        assert len(other) == len(got[0])
        for p, q in zip(got[0], other):
            assert np.array_equal(p, q)


def test_products_give_their_memory_back():
    """120 B per point and 32 B per edge of the plan and the incoming edges, 1056 B per
    point of the stages' forwards (limited, K = 3), 16 B per edge of the context."""
    import torch

    from paper_2403_13287_gb300.lskum import Solver
    c = naca0012_cloud(512, 311, seed=3)
    U = torch.from_numpy(smooth_state(c, 0.85, 1.0, amp=0.05, seed=9)).cuda()
    bar = torch.ones_like(U)
    s = Solver(c, order=2, inner_iters=3, time_scheme=1, limiter_K=1.0, mach=0.85, aoa_deg=1.0, reorder=1)
    s.step_vjp(bar, U=U)
    torch.cuda.empty_cache()
    free0 = torch.cuda.mem_get_info()[0]
    s.set_lean()
    given = torch.cuda.mem_get_info()[0] - free0
    s.close()
    want = (120 + 1056) * c["n"] + (32 + 16) * c["nbr_idx"].size
    assert abs(given - want) <= 8 << 20, (given, want)
