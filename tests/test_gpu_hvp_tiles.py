"""The optimisers' Hessian products over several tiles of perturbations (a tile holds
47 rows of 64 dims, 236 of 12): one row short of a tile, one more, a short last tile and
the most perturbations, each product against the oracle's estimate of it."""
import numpy as np
import pytest

import oracle as O
from paper_2412_03489_gb300 import build as hb
from paper_2412_03489_gb300 import hr
from paper_2412_03489_gb300 import workloads as wl
from parity import assert_estimate_close

pytestmark = pytest.mark.gpu

hb.build()

SIZES = [(64, 46), (64, 48), (64, 94), (64, 96), (64, 512), (12, 236), (12, 238), (12, 512)]


def scene(n):
    return wl.tris2d_scene(width=24, height=20, n_tris=max(2, n // 6), n_params=n, n_instances=2)


@pytest.mark.parametrize("n,M", SIZES)
def test_newton_cg_products(n, M):
    sc = scene(n)
    S, r, B, K = hr.Scene(sc), O.Tris2dRenderer(sc), 2, 2
    o = hr.hr_cg_opts()
    o.sigma, o.n_grad, o.n_hvp, o.cg_iters = sc["sigma"], 8, M, K
    o.lambda_rel, o.trust_radius, o.seed, o.request_base = 1e-3, 0.05, 99, 10
    th = np.ascontiguousarray(sc["theta_init"][:B], np.float64)
    st = hr.hr_optstate_create(S.handle, B, th, o)
    info = (hr.hr_step_info * B)()
    hr.hr_newton_cg_step(S.handle, st, info)
    _, p, hp = hr.hr_optstate_trace(st, B, K, n)
    hr.hr_optstate_destroy(st)
    S.close()
    for b in range(B):
        assert info[b].iters >= 1
        for i in range(info[b].iters):
            ref = O.estimate(r, "hvp", th[b], sc["sigma"], M, "aggregate", 99, 10 + b, sub=1 + i, v=p[b, i])
            assert_estimate_close(hp[b, i], ref, what=f"instance {b} product {i}")


@pytest.mark.parametrize("n,M", SIZES)
def test_published_optimisers_products(n, M):
    sc = scene(n)
    S, r, B = hr.Scene(sc), O.Tris2dRenderer(sc), 2
    o = hr.hr_ncg_opts()
    for k, v in dict(sigma_start=0.02, sigma_end=0.01, anneal_iters=4, n_grad=8, n_hvp=M, ls_iters=2, ls_tol=1e-4,
                     recompute=3, residual_mode=0, trust_radius=0.05, lambda_rel=1e-3, seed=99, request_base=10,
                     use_graph=0).items():
        setattr(o, k, v)
    x = np.ascontiguousarray(sc["theta_init"][:B], np.float64)
    st = hr.hr_ncg_create(S.handle, B, x, o)
    info = (hr.hr_ncg_info * B)()
    hr.hr_ncg_run(S.handle, st, 1, info)
    _, d, hd = hr.hr_ncg_trace(st, B, n)
    hr.hr_ncg_destroy(st)
    S.close()
    for b in range(B):
        ref = O.estimate(r, "hvp", x[b], info[b].sigma, M, "aggregate", 99, 10 + b, sub=1, v=d[b])
        assert_estimate_close(hd[b], ref, what=f"instance {b}")
