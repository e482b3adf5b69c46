"""Disc mismatch counts by rows (two exact tests per span end, the target's ones
counted by column) against the oracle's per-pixel counts, at the shapes and
positions where a span's ends leave the common case, for the plain kernel (a
render per warp) and the persistent queue (a render per lane)."""
import numpy as np
import pytest

import oracle as O
from paper_2412_03489_gb300 import build as hb
from paper_2412_03489_gb300 import hr
from paper_2412_03489_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

hb.build()


@pytest.mark.parametrize("size", [(1, 1), (1, 40), (31, 33), (32, 32), (65, 64), (97, 2), (1024, 5), (5, 1024)])
@pytest.mark.parametrize("radius,sigma", [(0.2, 0.05), (0.004, 0.05), (0.7, 0.3), (30.0, 2.0), (0.25, 1e-7)])
def test_losses_and_queue(size, radius, sigma):
    W, H = size
    sc = wl.disc_scene(seed=5, width=W, height=H, radius=radius)
    # the centre on a pixel centre: with a small sigma the edge passes within rounding of others
    th = np.array([(W // 2 + 0.5) / W, (H // 2 + 0.5) / H])
    target = (np.random.default_rng(W + H).random(W * H) < 0.5).astype(np.float32)
    S, r, M = hr.Scene(sc, target), O.DiscRenderer(sc, target), 70
    out, d = S.estimate(hr.HR_HESSIAN, th, sigma, M, hr.HR_AGGREGATE, 3, 4, debug=True)
    want = np.array([r.loss(th.astype(np.float32) + t, None) for t in d["tau"]]).astype(np.float32)
    assert np.array_equal(d["losses"], want)
    q = hr.hr_queue_create(S, max_requests=4, idle_budget_us=200)
    got = np.zeros((2, 2))
    hr.hr_queue_wait(q, hr.hr_queue_submit(q, hr.HR_HESSIAN, th, None, hr.make_opts(sigma, M, hr.HR_AGGREGATE, 3, 4)), got)
    hr.hr_queue_destroy(q)
    assert np.array_equal(got, out)
    S.close()
