"""Mesh losses against the oracle where the tiles' edge cases lie: the target is
read in tile order (8x4 and 8x8 tiles, padded with zeros), so images whose width
or height leaves a partial tile, or is smaller than one, are compared loss by loss."""
import numpy as np
import pytest

import oracle as O
from paper_2412_03489_gb300 import build as hb
from paper_2412_03489_gb300 import hr
from paper_2412_03489_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

hb.build()


@pytest.mark.parametrize("size", [(1, 1), (3, 9), (8, 4), (9, 5), (33, 31), (64, 50), (390, 403), (401, 389)])
def test_losses(size):
    W, H = size
    sc = wl.revolve_scene(width=W, height=H)
    target = np.random.default_rng(W * H).random((H * W * 3)).astype(np.float32)   # no zero pixel, also outside the mesh
    S, r = hr.Scene(sc, target), O.RevolveRenderer(sc, target=target)
    th = np.asarray(sc["theta_query"], np.float64)
    _, d = S.estimate(hr.HR_HESSIAN, th, 0.3, 6, hr.HR_AGGREGATE, 3, 4, debug=True)
    S.close()
    want = np.array([r.loss(th.astype(np.float32) + t, None) for t in d["tau"]])
    # FP32 squares, all positive, in sequential sums of at most 192 terms (a tile that
    # nothing covers), then trees: under 230 units of 2^-24, and shades of a few
    # units each, twice in a square: 2e-5 in all
    np.testing.assert_allclose(d["losses"], want, rtol=2e-5)


def test_a_smaller_scene_made_later_leaves_a_larger_one_its_launches():
    """The kernels' shared-memory limits are the process's: a scene with a small
    layout made after one with a large layout does not lower them."""
    big, th = wl.revolve_scene(width=512, height=512), np.asarray(wl.revolve_scene()["theta_query"], np.float64)
    mid = wl.revolve_scene(width=64, height=64)
    scenes = [hr.Scene(sc) for sc in (big, mid)]
    before = [S.estimate(hr.HR_HESSIAN, th, 0.1, 4, hr.HR_AGGREGATE, 3, 4) for S in scenes]
    small = dict(mid, width=8, height=8)
    small["vertices"], small["triangles"] = wl.sheets_mesh(layers=1, grid=1)
    late = hr.Scene(small)
    after = [S.estimate(hr.HR_HESSIAN, th, 0.1, 4, hr.HR_AGGREGATE, 3, 4) for S in scenes]
    for S in scenes + [late]:
        S.close()
    assert all(np.array_equal(a, b) for a, b in zip(after, before))


@pytest.mark.parametrize("layers,grid,size", [(8, 8, 128), (8, 8, 256), (14, 8, 256), (8, 8, 512), (14, 8, 512), (12, 4, 300)])
def test_stacked_sheets(layers, grid, size):
    """Every triangle faces the camera and every tile is many layers deep: bins filled at
    once, in a few bands of tile rows and in many, loss by loss (tolerance as above)."""
    sc = wl.revolve_scene(width=size, height=size)
    sc["vertices"], sc["triangles"] = wl.sheets_mesh(layers, grid)
    S, r = hr.Scene(sc), O.RevolveRenderer(sc)
    th = np.asarray(sc["theta_query"], np.float64)
    _, d = S.estimate(hr.HR_HESSIAN, th, 0.1, 4, hr.HR_AGGREGATE, 3, 4, debug=True)
    S.close()
    want = np.array([r.loss(th.astype(np.float32) + t, None) for t in d["tau"]])
    np.testing.assert_allclose(d["losses"], want, rtol=2e-5)
