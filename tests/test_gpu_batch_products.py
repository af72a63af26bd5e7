"""A cloud's products are the same bits alone and inside a batch: no reverse
kernel adds in an order that depends on the number of points (needs a GPU)."""
import numpy as np
import pytest

from paper_2403_13287_gb300.cloudgen import naca0012_cloud, smooth_state

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order,limiter,gamma,reorder", [(2, 0.0, 1.4, 1), (2, 1.0, 1.4, 0), (2, 0.0, 1.3, 1), (1, 0.0, 1.4, 1)])
def test_products_of_a_cloud_do_not_depend_on_the_batch(order, limiter, gamma, reorder):
    """3250 points alone and beside 64k points: residual and step products, all of
    U_bar, x_bar and y_bar."""
    import torch

    from paper_2403_13287_gb300.lskum import Solver
    a, big = naca0012_cloud(130, 24, seed=11), naca0012_cloud(324, 197, seed=4)
    n = a["n"]
    kw = dict(order=order, inner_iters=3 if order == 2 else 0, time_scheme=1, limiter_K=limiter, precision=0,
              reorder=reorder, gamma=gamma)
    U0 = [smooth_state(c, 0.85, 1.0, amp=0.05, seed=9, gamma=gamma) for c in (a, big)]
    Rb = np.random.default_rng(2).standard_normal((4, n + big["n"]))
    got = []
    for clouds in ([a], [a, big]):
        m = sum(c["n"] for c in clouds)
        s = Solver.batch([(c, 0.85, 1.0) for c in clouds], **kw) if len(clouds) > 1 else Solver(a, mach=0.85, aoa_deg=1.0, **kw)
        U = torch.from_numpy(np.ascontiguousarray(np.concatenate(U0[:len(clouds)], axis=1))).cuda()
        bar = torch.from_numpy(np.ascontiguousarray(Rb[:, :m])).cuda()
        out = s.residual_vjp(bar, U) + s.step_vjp(bar, U=U)
        got.append([t.cpu().numpy()[..., :n] for t in out])
        s.close()
    for name, p, q in zip(("U_bar", "x_bar", "y_bar", "step U_bar", "step x_bar", "step y_bar"), *got):
        assert np.array_equal(p, q), name
