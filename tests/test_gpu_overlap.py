"""Estimates issued one after another on a stream without waiting, whose kernels
overlap: the sampler of one call runs beside the last kernels of the call before, in the
same workspace.  Every result equals the one of the same call made alone."""
import numpy as np
import pytest
import torch

from paper_2412_03489_gb300 import build as hb
from paper_2412_03489_gb300 import hr
from paper_2412_03489_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

hb.build()

SCENES = {
    "disc": lambda: wl.disc_scene(width=40, height=33),
    "disc large": lambda: wl.disc_scene(width=333, height=250),
    "squares": lambda: wl.boxes_scene(5, seed=3),
    "tris": lambda: wl.tris2d_scene(seed=3, width=64, height=48, n_tris=8, n_params=20),
    "mesh": lambda: wl.revolve_scene(width=64, height=64),
    "mesh without a compact layout": lambda: wl.revolve_scene(width=400, height=390),
    "path-traced": lambda: wl.ptbox_scene(width=32, height=32, spp=1, target_spp=2),
    "quadratic": lambda: wl.quadratic_scene(A=np.eye(3), b=np.ones(3), theta=np.zeros(3), sigma=0.1),
}


@pytest.mark.parametrize("name", list(SCENES))
@pytest.mark.parametrize("entry", [hr.hr_estimate_dev, hr.hr_estimate_dev_noalloc])
def test_calls_in_a_row(name, entry):
    sc = SCENES[name]()
    S, n = hr.Scene(sc), sc["n_params"]
    g = np.random.default_rng(1)
    calls = []
    for k in range(24):
        q, strategy = k % 3, hr.HR_AGGREGATE if k % 2 or n > 10 else hr.HR_ELEMENTWISE
        M = int(g.choice([2, 34, 256])) if "400" not in str(sc["width"]) else 34
        o = hr.make_opts(sc["sigma"], M, strategy, 3 + k, k, stream=torch.cuda.current_stream().cuda_stream or 1)
        theta = torch.tensor(np.asarray(sc["theta_query"]) + g.normal(0, 0.02, n), device="cuda")
        v = torch.tensor(g.normal(size=n), device="cuda")
        calls.append((q, o, theta, v))

    def run(wait):
        outs, th, v = [], torch.zeros(n, dtype=torch.float64, device="cuda"), torch.zeros(n, dtype=torch.float64, device="cuda")
        for q, o, theta, vv in calls:
            out = torch.full((n, n) if q == hr.HR_HESSIAN else (n,), float("nan"), dtype=torch.float64, device="cuda")
            th.copy_(theta)   # the inputs written, and the results used, on the stream
            v.copy_(vv)
            entry(S.handle, q, th.data_ptr(), v.data_ptr() if q == hr.HR_HVP else None, o, out.data_ptr())
            outs.append(out * 2.0)
            if wait:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        return [x.cpu().numpy() for x in outs]

    def bare(repeat):   # nothing between the calls but the calls
        outs = [torch.full((n, n) if q == hr.HR_HESSIAN else (n,), float("nan"), dtype=torch.float64, device="cuda")
                for q, *_ in calls]
        torch.cuda.synchronize()
        for _ in range(repeat):
            for (q, o, theta, v), out in zip(calls, outs):
                entry(S.handle, q, theta.data_ptr(), v.data_ptr() if q == hr.HR_HVP else None, o, out.data_ptr())
        torch.cuda.synchronize()
        return [2.0 * x.cpu().numpy() for x in outs]

    want = run(True)
    assert all(np.isfinite(x).all() for x in want)
    for got in (run(False), bare(1), bare(5)):
        assert all(np.array_equal(a, b) for a, b in zip(got, want))
    S.close()


@pytest.mark.parametrize("name", ["disc", "tris", "mesh", "path-traced"])
def test_captured_calls(name):
    """The no-allocation entry captured three times in a row into a graph (its first kernel has
    no kernel before it there) and replayed: the results of the calls made alone."""
    sc = SCENES[name]()
    S, n = hr.Scene(sc), sc["n_params"]
    theta = torch.tensor(np.asarray(sc["theta_query"], np.float64), device="cuda")
    outs = [torch.zeros((n, n), dtype=torch.float64, device="cuda") for _ in range(3)]

    def calls(stream):
        for k, out in enumerate(outs):
            o = hr.make_opts(sc["sigma"], 34, hr.HR_AGGREGATE, 3 + k, k, stream=stream.cuda_stream)
            hr.hr_estimate_dev_noalloc(S.handle, hr.HR_HESSIAN, theta.data_ptr(), None, o, out.data_ptr())

    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        calls(side)
    torch.cuda.synchronize()
    want = [x.cpu().numpy().copy() for x in outs]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        calls(side)
    for _ in range(3):
        for x in outs:
            x.zero_()
        graph.replay()
    torch.cuda.synchronize()
    assert all(np.array_equal(x.cpu().numpy(), w) for x, w in zip(outs, want))
    S.close()
