"""The path tracer's pair kernel (both legs of an antithetic pair by one block
or one cluster) against the kernel that renders one perturbation per block,
which the counting build always runs: the same bits, at the sizes where the
launch changes between them and between whole pairs and clusters, at ragged
pixel counts, and where paths leave the common case (light near or beyond the
walls, legs that end on the light, deep paths, a large sphere 0)."""
import numpy as np
import pytest

from paper_2412_03489_gb300 import build as hb
from paper_2412_03489_gb300 import hr
from paper_2412_03489_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

hb.build()


def losses(S, sc, M, sigma, strategy, count):
    hr.hr_scene_count_work(S.handle, count)
    v = np.ones(6)
    _, d = S.estimate(hr.HR_HVP, np.asarray(sc["theta_query"]), sigma, M, strategy, 5, 6, 7, v=v, debug=True)
    return d["losses"]


@pytest.mark.parametrize("shape", [
    # width, height, spp, renders
    (31, 33, 2, 60), (32, 32, 1, 64), (33, 32, 2, 130), (32, 32, 1, 2000), (47, 49, 1, 128), (48, 48, 1, 400),
    (64, 64, 1, 2), (64, 63, 2, 200), (65, 64, 1, 1000), (64, 64, 1, 5200), (128, 97, 1, 40), (300, 7, 3, 30),
])
@pytest.mark.parametrize("strategy", [hr.HR_AGGREGATE, hr.HR_PLAIN])
def test_pairs_equal_single_renders(shape, strategy):
    W, H, spp, M = shape
    sc = wl.ptbox_scene(seed=40, width=W, height=H, spp=spp, target_spp=2)
    S = hr.Scene(sc)
    assert np.array_equal(losses(S, sc, M, 0.05, strategy, False), losses(S, sc, M, 0.05, strategy, True))
    S.close()


@pytest.mark.parametrize("what", ["wide", "light_high", "big_sphere", "deep", "depth1", "camera_outside", "many_samples"])
def test_pairs_equal_single_renders_off_the_common_path(what):
    sc = wl.ptbox_scene(seed=41, width=40, height=36, spp=2, target_spp=2)
    sigma = 0.4 if what == "wide" else 0.05
    if what == "light_high":
        sc["theta_query"] = np.array(sc["theta_query"])
        sc["theta_query"][1] = 0.98
    elif what == "big_sphere":
        sc["sph_radius"] = np.array([0.7, 0.2, 0.15], np.float32)
    elif what == "deep":
        sc["depth"] = 15
    elif what == "depth1":
        sc["depth"] = 1
    elif what == "camera_outside":
        sc["cam_z"] = np.float32(1.4)
    elif what == "many_samples":
        sc["spp"] = 37
    S = hr.Scene(sc)
    assert np.array_equal(losses(S, sc, 70, sigma, hr.HR_AGGREGATE, False),
                          losses(S, sc, 70, sigma, hr.HR_AGGREGATE, True))
    S.close()
