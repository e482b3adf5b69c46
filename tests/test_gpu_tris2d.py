"""The coloured-triangle loss kernel against the oracle's per-pixel edge tests
at the sizes where its column spans, 8x4 tiles, 32-row bands and renders per
CTA have edges."""
import numpy as np
import pytest

import oracle as O
from paper_2412_03489_gb300 import build as hb
from paper_2412_03489_gb300 import hr
from paper_2412_03489_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

hb.build()


def check(sc, M, compare, sigma):
    """The losses of `compare` of the M renders against the oracle.  The kernel
    sums npx / 256 squared colour differences per lane in FP32 (four roundings
    each), then 5 shuffle and 8 warp sums: at most npx / 256 + 24 roundings of
    2^-24 relative to the sum of non-negative terms."""
    S, r = hr.Scene(sc), O.Tris2dRenderer(sc)
    th = np.asarray(sc["theta_query"], np.float64)
    _, d = S.estimate(hr.HR_GRAD, th, sigma, M, hr.HR_AGGREGATE, 3, 4, debug=True)
    tol = (sc["width"] * sc["height"] / 256 + 24) * 2.0 ** -24
    for m in compare:
        ref = r.loss(th.astype(np.float32) + d["tau"][m])
        assert abs(d["losses"][m] - ref) <= tol * ref, (m, d["losses"][m], ref)
    S.close()
    return d["losses"]


@pytest.mark.parametrize("sigma", [0.02, 1.0])
@pytest.mark.parametrize("size", [(1, 1), (7, 3), (8, 4), (9, 33), (64, 32), (65, 31), (520, 36), (36, 520)])
@pytest.mark.parametrize("n_tris", [1, 16, 32])
def test_losses_at_tile_and_band_edges(size, n_tris, sigma):
    sc = wl.tris2d_scene(seed=31, width=size[0], height=size[1], n_tris=n_tris, n_params=9, n_instances=1)
    check(sc, 10, range(10), sigma)


@pytest.mark.parametrize("sigma", [1e-7, 1e-3])
def test_losses_with_edges_on_pixel_centres(sigma):
    """Vertices on a 1/128 grid of a 64x64 image: edges through pixel centres
    (E = 0), axis-aligned and diagonal edges, shared edges, a triangle of
    no area."""
    sc = wl.tris2d_scene(seed=9, width=64, height=64, n_tris=8, n_params=9, n_instances=1)
    raw = np.array(sc["raw_params"]).reshape(8, 9)
    raw[:, :6] = np.random.default_rng(3).integers(0, 129, (8, 6)) / 128.0
    raw[3, :6] = raw[2, [0, 1, 4, 5, 2, 3]]
    raw[4, :6] = [0, 0, 1, 0, 1, 1]
    raw[5, :6] = [0, 0, 1, 1, 0, 1]
    raw[6, :6] = [0.5, 0.5, 0.5, 0.5, 0.2, 0.2]
    sc["raw_params"], sc["param_index"] = raw.reshape(-1).astype(np.float32), np.arange(63, 72, dtype=np.int32)
    sc["theta_target"] = sc["theta_query"] = raw.reshape(-1)[63:].astype(np.float64)
    check(sc, 64, range(64), sigma)


def test_renders_per_cta_do_not_change_losses():
    """One, two and four renders per CTA (the last CTA partly filled): pair k
    draws the same perturbations whatever M, so the losses are the same bits."""
    sc = wl.tris2d_scene(seed=8, width=40, height=37, n_instances=1)
    one = check(sc, 512, (0, 511), 0.02)
    for M in (1502, 3002):
        many = check(sc, M, (0, M - 1), 0.02)
        assert np.array_equal(many[:512], one)
        assert np.array_equal(check(sc, 3006, (3005,), 0.02)[:M], many)
