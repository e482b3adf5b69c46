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


@pytest.mark.parametrize("size", [(1, 1), (7, 40), (31, 33), (32, 5), (64, 64), (65, 64), (333, 20), (512, 9), (1024, 5), (5, 1024)])
def test_grey_targets(size):
    """Targets with values other than 0 and 1: every launch shape and the queue give the same
    bits, and the losses are the mean square difference to within its FP32 sum's
    rounding (npx / 32 + 5 additions and a division, 2^-24 each)."""
    W, H = size
    sc = wl.disc_scene(seed=5, width=W, height=H, radius=0.3)
    target = np.random.default_rng(W + H).uniform(-0.5, 1.5, W * H).astype(np.float32)
    S, M, th = hr.Scene(sc, target), 34, np.asarray(sc["theta_query"], np.float64)
    out, d = S.estimate(hr.HR_HESSIAN, th, 0.1, M, hr.HR_AGGREGATE, 3, 4, debug=True)
    f32 = np.float32
    px, py = (np.arange(W, dtype=f32) + f32(0.5)) / f32(W), (np.arange(H, dtype=f32) + f32(0.5)) / f32(H)
    c = th.astype(f32) + d["tau"]
    dx, dy = px[None, :] - c[:, :1], py[None, :] - c[:, 1:]
    # fma(dx, dx, dy^2): one rounding of the sum, whose terms FP64 holds
    d2 = ((dx.astype(np.float64) ** 2)[:, None, :] + (dy * dy).astype(np.float64)[:, :, None]).astype(f32)
    inside = d2 < f32(sc["radius"]) * f32(sc["radius"])
    diff = inside.reshape(M, -1).astype(f32) - target
    want = (diff.astype(np.float64) ** 2).mean(1)
    assert np.all(np.abs(d["losses"] - want) <= (W * H / 32 + 7) * 2.0 ** -24 * want)
    for variant in (1, 2):
        hr.hr_set_tuning(S.handle, variant, 32)
        assert np.array_equal(S.estimate(hr.HR_HESSIAN, th, 0.1, M, hr.HR_AGGREGATE, 3, 4), out)
    q = hr.hr_queue_create(S, max_requests=4, idle_budget_us=200)
    got = np.zeros((2, 2))
    hr.hr_queue_wait(q, hr.hr_queue_submit(q, hr.HR_HESSIAN, th, None, hr.make_opts(0.1, M, hr.HR_AGGREGATE, 3, 4)), got)
    hr.hr_queue_destroy(q)
    assert np.array_equal(got, out)
    S.close()
