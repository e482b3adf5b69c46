"""The measured work of this framework: what a user has it do, through its public entry points.

Every case is an estimate (gradient, Hessian or Hessian-vector product of a smoothed rendering loss)
of one of the renderers, a step of one of the two optimisers, a batch of requests through the
persistent queue, or a burst of mixed requests through the server.  Scenes, sizes and options are
those of the package's seeded workloads, of its tests and of its benchmark, or generic ones of the
same ranges.  `exact` restates the method in 64 bits with torch: the random draws are the ones the
library documents (Philox4x32-10 counters, perturbations rounded once to 32 bits), everything after
them is plain 64-bit arithmetic.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2412_03489_gb300 import hr
from paper_2412_03489_gb300 import workloads as wl

QUANTITY = {"grad": hr.HR_GRAD, "hessian": hr.HR_HESSIAN, "hvp": hr.HR_HVP}
STRATEGY = {"elementwise": hr.HR_ELEMENTWISE, "aggregate": hr.HR_AGGREGATE}
LEGACY_STREAM = 1   # cudaStreamLegacy: torch's default stream, so that results are ordered with torch's work
F64 = torch.float64
DEV = "cuda" if torch.cuda.is_available() else "cpu"


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def _estimate(scene, width, height, quantity, strategy, samples, **more):
    return dict(kind="estimate", scene=scene, width=width, height=height, quantity=quantity, strategy=strategy,
                samples=samples, host=False, **more)


def listed():
    return [
        # the smallest call: one element-wise 2x2 Hessian of a disc, as an optimisation loop on a
        # plateau task issues it, on device pointers
        dict(_estimate("disc", 64, 64, "hessian", "elementwise", 1024), name="disc_hessian"),
        # many samples of a larger image with odd sides (one aggregate estimate near convergence)
        dict(_estimate("disc", 333, 250, "hessian", "aggregate", 16384), name="disc_ragged_hessian"),
        # five squares, ten parameters, all 55 elements of the Hessian with samples of their own,
        # through the host-array entry point (the variance study's call)
        dict(_estimate("squares", 64, 64, "hessian", "elementwise", 64, squares=5) | dict(host=True),
             name="squares_hessian_host"),
        # the benchmark's configuration: 2,048-triangle mesh, 256x256, 4,096 renders
        dict(_estimate("mesh", 256, 256, "hessian", "aggregate", 4096, rings=33, slices=32), name="mesh_hessian"),
        # the largest mesh image with few samples (the serving mix's 512x512 request)
        dict(_estimate("mesh", 512, 512, "hessian", "aggregate", 256, rings=33, slices=32), name="mesh_large_image"),
        # the path-traced box at the benchmark's size: the largest call
        dict(_estimate("ptbox", 128, 128, "hvp", "aggregate", 8192, spp=4), name="ptbox_hvp"),
        # the serving mix's small path-traced request: too few renders to fill the GPU by number alone
        dict(_estimate("ptbox", 64, 64, "hvp", "aggregate", 256, spp=2), name="ptbox_small_hvp"),
        # the full 64x64 Hessian of a triangle scene from 1,024 renders (2,080 unique elements)
        dict(_estimate("tris", 128, 128, "hessian", "aggregate", 1024, n_params=64, n_tris=16), name="tris_hessian"),
        # one Newton-CG step of 64 instances, 64 parameters, 10 CG iterations, replayed as a graph
        dict(kind="newton", width=256, height=256, n_params=64, n_tris=16, instances=64, n_grad=32, n_hvp=32,
             cg_iters=10, name="tris_newton_step"),
        # two evaluations of the published optimiser on the mesh, 64 instances, 256 + 256 renders each
        dict(kind="optimise", width=128, height=128, rings=33, slices=32, instances=64, n_grad=256, n_hvp=256,
             evals=2, name="mesh_optimise"),
        # 512 disc Hessians through the persistent queue, host arrays to host results
        dict(kind="queue", width=64, height=64, samples=1024, requests=512, name="queue_disc"),
        # a burst of 48 mixed estimates on seven resident scenes through the continuous-batching server
        dict(kind="serve", requests=48, name="serve_burst"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _even(x, lo=2):
    return max(lo, int(x) & ~1)


def draw(rng):
    kind = rng.choice(["disc", "disc", "squares", "mesh", "mesh", "ptbox", "tris", "tris", "newton", "optimise", "queue"])
    if kind == "disc":
        return _estimate("disc", _log_int(rng, 24, 700), _log_int(rng, 24, 700), rng.choice(["grad", "hessian", "hvp"]),
                         rng.choice(["elementwise", "aggregate"]), _even(_log_int(rng, 128, 16384))) | \
            dict(host=rng.random() < 0.3)
    if kind == "squares":
        k = rng.randint(1, 6)
        q = rng.choice(["grad", "hessian", "hvp"])
        s = rng.choice(["elementwise", "aggregate"])
        groups = (k * (2 * k + 1) if q == "hessian" else 2 * k) if s == "elementwise" else 1
        return _estimate("squares", _log_int(rng, 24, 300), _log_int(rng, 24, 300), q, s,
                         _even(_log_int(rng, 512, 16384) / groups), squares=k) | dict(host=rng.random() < 0.3)
    if kind == "mesh":
        w, h = _log_int(rng, 48, 512), _log_int(rng, 48, 512)
        return _estimate("mesh", w, h, rng.choice(["grad", "hessian", "hvp"]), rng.choice(["elementwise", "aggregate"]),
                         _even(min(_log_int(rng, 64, 4096), 3.2e7 / (w * h)) if w * h > 1 << 16 else _log_int(rng, 64, 2048)),
                         rings=rng.randint(9, 33), slices=rng.randint(8, 32))
    if kind == "ptbox":
        w, h, spp = _log_int(rng, 24, 128), _log_int(rng, 24, 128), rng.randint(1, 4)
        return _estimate("ptbox", w, h, rng.choice(["grad", "hvp"]), "aggregate",
                         _even(min(_log_int(rng, 64, 8192), 2.5e8 / (w * h * spp))), spp=spp)
    if kind == "tris":
        n_tris = rng.randint(4, 32)
        w, h = _log_int(rng, 48, 400), _log_int(rng, 48, 400)
        return _estimate("tris", w, h, rng.choice(["grad", "hessian", "hvp"]), "aggregate",
                         _even(min(_log_int(rng, 64, 4096), 2e8 / (w * h))),
                         n_params=rng.randint(4, min(64, 9 * n_tris)), n_tris=n_tris)
    if kind == "newton":
        return dict(kind="newton", width=_log_int(rng, 48, 256), height=_log_int(rng, 48, 256),
                    n_params=rng.randint(8, 64), n_tris=rng.randint(8, 24), instances=_log_int(rng, 1, 64),
                    n_grad=_even(rng.randint(16, 64)), n_hvp=_even(rng.randint(16, 64)), cg_iters=rng.randint(2, 10))
    if kind == "optimise":
        return dict(kind="optimise", width=_log_int(rng, 48, 256), height=_log_int(rng, 48, 256),
                    rings=rng.randint(9, 33), slices=rng.randint(8, 32), instances=_log_int(rng, 1, 32),
                    n_grad=_even(_log_int(rng, 32, 256)), n_hvp=_even(_log_int(rng, 32, 256)), evals=rng.randint(1, 3))
    return dict(kind="queue", width=_log_int(rng, 32, 256), height=_log_int(rng, 32, 256),
                samples=_even(_log_int(rng, 64, 1024)), requests=_log_int(rng, 64, 512))


# ---------------------------------------------------------------------------
# what a user's program has in hand
# ---------------------------------------------------------------------------
def _scene_dict(case, seed):
    w, h = case["width"], case["height"]
    scene = case.get("scene", {"newton": "tris", "optimise": "mesh", "queue": "disc"}.get(case["kind"]))
    if scene == "disc":
        return wl.disc_scene(seed=seed, width=w, height=h)
    if scene == "squares":
        return wl.boxes_scene(case["squares"], seed=seed, width=w, height=h)
    if scene == "mesh":
        sc = wl.revolve_scene(seed=seed, width=w, height=h)
        if (case["rings"], case["slices"]) != (33, 32):
            radii = np.random.default_rng(seed).uniform(0.3, 0.8, size=8)
            sc["vertices"], sc["triangles"] = wl.revolve_mesh(radii, case["rings"], case["slices"])
        return sc
    if scene == "ptbox":
        return wl.ptbox_scene(seed=seed, width=w, height=h, spp=case["spp"])
    return wl.tris2d_scene(seed=seed, width=w, height=h, n_tris=case["n_tris"], n_params=case["n_params"],
                           n_instances=case.get("instances", 1))


def _direction(sc, seed):
    return np.random.default_rng(seed + 1).normal(size=sc["n_params"])


_KEPT = {}   # the queue and the server that a serving program keeps open between batches


def _optimise_inputs(case, seed):
    sc = _scene_dict(case, seed)
    th0 = np.asarray(sc["theta_target"]) + np.random.default_rng(seed + 2).normal(0.0, 0.1, (case["instances"], 2))
    return sc, np.ascontiguousarray(th0)


def _queue_inputs(case, seed):
    sc = _scene_dict(case, wl.disc_scene()["seed"])
    g = np.random.default_rng(seed)
    thetas = np.asarray(sc["theta_query"]) + g.normal(0.0, 0.01, (case["requests"], 2))
    return sc, thetas, g.integers(1, 1 << 40, case["requests"])


def _serve_inputs(case, seed):
    """The serving workload's scenes and its estimate requests (every kind of them, none of the steps)."""
    scenes = wl.serving_scenes()
    kinds = [k for k in wl.SERVING_KINDS if k[1] != hr.HR_NEWTON_STEP]
    g = np.random.default_rng(seed)
    reqs = []
    for i in range(case["requests"]):
        name, q, strategy, samples = kinds[(5 * i) % len(kinds)]
        sc = scenes[name]
        n = sc["n_params"]
        reqs.append(dict(scene=name, quantity=q, strategy=strategy, M=samples, sigma=sc["sigma"],
                         theta=np.asarray(sc["theta_query"]) + g.normal(0.0, 0.01, n), v=g.normal(size=n),
                         seed=int(g.integers(1, 1 << 40)), request=i))
    return scenes, reqs


def prepare(case, seed):
    kind = case["kind"]
    if kind == "estimate":
        sc = _scene_dict(case, seed)
        s = hr.Scene(sc)
        n, q = s.n, QUANTITY[case["quantity"]]
        v = _direction(sc, seed) if q == hr.HR_HVP else None
        state = dict(kind="host" if case["host"] else "dev", scene=s, q=q, sigma=sc["sigma"], M=case["samples"],
                     strategy=STRATEGY[case["strategy"]], seed=seed, theta=np.asarray(sc["theta_query"], np.float64), v=v)
        if not case["host"]:
            state["opts"] = hr.make_opts(sc["sigma"], case["samples"], state["strategy"], seed, 0, stream=LEGACY_STREAM)
            state["d_theta"] = torch.tensor(state["theta"], dtype=F64, device="cuda")
            state["d_v"] = None if v is None else torch.tensor(v, dtype=F64, device="cuda")
            state["out"] = torch.zeros((n, n) if q == hr.HR_HESSIAN else (n,), dtype=F64, device="cuda")
        return state
    if kind == "newton":
        sc = _scene_dict(case, seed)
        s = hr.Scene(sc)
        o = hr.hr_cg_opts()
        o.sigma, o.n_grad, o.n_hvp, o.cg_iters = sc["sigma"], case["n_grad"], case["n_hvp"], case["cg_iters"]
        o.lambda_rel, o.trust_radius, o.seed, o.request_base, o.use_graph = 1e-3, 0.05, seed, 0, 1
        b = case["instances"]
        st = hr.hr_optstate_create(s.handle, b, np.ascontiguousarray(sc["theta_init"]), o)
        return dict(kind=kind, st=_Owned(st, hr.hr_optstate_destroy), scene=s, info=(hr.hr_step_info * b)(), B=b, n=s.n)
    if kind == "optimise":
        sc, th0 = _optimise_inputs(case, seed)
        s = hr.Scene(sc)
        o = hr.hr_ncg_opts()
        for k, x in _optimiser_options(case, seed).items():
            setattr(o, k, x)
        b, e = case["instances"], case["evals"]
        st = hr.hr_ncg_create(s.handle, b, th0, o)
        return dict(kind=kind, st=_Owned(st, hr.hr_ncg_destroy), scene=s, info=(hr.hr_ncg_info * (b * e))(), B=b, evals=e)
    if kind == "queue":
        sc, thetas, seeds = _queue_inputs(case, seed)
        key = ("queue", case["width"], case["height"])
        if key not in _KEPT:
            s = hr.Scene(sc)
            _KEPT[key] = (s, hr.hr_queue_create(s, max_requests=1024, idle_budget_us=1000))
        opts = hr.opts_array(sc["sigma"], case["samples"], hr.HR_ELEMENTWISE, seeds, range(len(seeds)))
        return dict(kind=kind, queue=_KEPT[key][1], thetas=thetas, opts=opts, out=np.zeros((len(seeds), 2, 2)))
    scenes, reqs = _serve_inputs(case, seed)
    if "serve" not in _KEPT:
        _KEPT["serve"] = ({k: hr.Scene(v) for k, v in scenes.items()}, hr.hr_server_create(256 << 20, max_active=32))
    resident, server = _KEPT["serve"]
    made = [hr.make_request(resident[r["scene"]], r["quantity"], r["theta"], r["v"] if r["quantity"] == hr.HR_HVP else None,
                            hr.make_opts(r["sigma"], r["M"], r["strategy"], r["seed"], r["request"])) for r in reqs]
    outs = [np.zeros((len(r["theta"]),) * (2 if r["quantity"] == hr.HR_HESSIAN else 1)) for r in reqs]
    return dict(kind=kind, server=server, made=made, outs=outs)


class _Owned:
    """An optimiser state, destroyed with the dict that holds it (which drops its values in order: before its scene)."""

    def __init__(self, handle, destroy):
        self.handle, self._destroy = handle, destroy

    def __del__(self):
        self._destroy(self.handle)


def run(state):
    kind = state["kind"]
    if kind == "dev":
        v = state["d_v"]
        hr.hr_estimate_dev(state["scene"].handle, state["q"], state["d_theta"].data_ptr(),
                           None if v is None else v.data_ptr(), state["opts"], state["out"].data_ptr())
        return state["out"]
    if kind == "host":
        return state["scene"].estimate(state["q"], state["theta"], state["sigma"], state["M"], state["strategy"],
                                       state["seed"], 0, v=state["v"])
    if kind == "newton":
        hr.hr_newton_cg_step(state["scene"].handle, state["st"].handle, state["info"])
        theta = np.zeros((state["B"], state["n"]))
        hr.hr_optstate_theta(state["st"].handle, theta)
        return dict(theta=theta, grad_norm=np.array([i.grad_norm for i in state["info"]]),
                    step_norm=np.array([i.step_norm for i in state["info"]]),
                    iters=np.array([i.iters for i in state["info"]]))
    if kind == "optimise":
        hr.hr_ncg_run(state["scene"].handle, state["st"].handle, state["evals"], state["info"])
        theta = np.zeros((state["B"], 2))
        hr.hr_ncg_theta(state["st"].handle, theta)
        return dict(theta=theta, grad_norm=np.array([i.grad_norm for i in state["info"]]),
                    alpha=np.array([i.alpha for i in state["info"]]))
    if kind == "queue":
        tickets = hr.hr_queue_submit_many(state["queue"], hr.HR_HESSIAN, state["thetas"], None, state["opts"])
        hr.hr_queue_wait_many(state["queue"], tickets, state["out"])
        return state["out"]
    info = hr.hr_request_info()
    tickets = [hr.hr_server_submit(state["server"], r) for r, _ in state["made"]]
    for t, out in zip(tickets, state["outs"]):
        hr.hr_server_wait(state["server"], t, out, info)
    return state["outs"]


# ---------------------------------------------------------------------------
# the work of one pass
# ---------------------------------------------------------------------------
def _render_flops(scene, w, h, verts=0, tris=0, spp=1, squares=0):
    """Operations that one render and its loss cannot do without, by the renderer's definition."""
    px = w * h
    if scene == "disc":
        return 6 * px                       # distance, compare, squared difference
    if scene == "squares":
        return (4 * squares + 3) * px
    if scene == "mesh":
        return 15 * verts + 40 * tris + 19 * px   # transform, set-up, one depth test and the colour difference a pixel
    if scene == "tris":
        return 19 * px
    return 950 * spp * px                   # about three hit rays, two and a half shadow rays and three vertices a path


def work(case):
    kind = case["kind"]
    if kind == "serve":
        scenes, reqs = _serve_inputs(case, 1)
        total = dict(bytes=0, flops=0)
        names = {wl.SCENE_DISC2D: "disc", wl.SCENE_REVOLVE3D: "mesh", wl.SCENE_PTBOX: "ptbox", wl.SCENE_TRIS2D: "tris"}
        for r in reqs:
            sc = scenes[r["scene"]]
            n = sc["n_params"]
            groups = n * (n + 1) // 2 if r["strategy"] == 0 else 1
            total["flops"] += groups * r["M"] * _render_flops(names[sc["kind"]], sc["width"], sc["height"],
                                                              len(sc.get("vertices", ())), len(sc.get("triangles", ())),
                                                              sc.get("spp", 1))
            total["bytes"] += 4 * sc["width"] * sc["height"] * sc["channels"] + 8 * (n + n * n)
        return total
    w, h = case["width"], case["height"]
    scene = case.get("scene", {"newton": "tris", "optimise": "mesh", "queue": "disc"}.get(kind))
    verts, tris = (case["rings"] * case["slices"], 2 * (case["rings"] - 1) * case["slices"]) if scene == "mesh" else (0, 0)
    n = {"disc": 2, "mesh": 2, "ptbox": 6}.get(scene) or (2 * case["squares"] if scene == "squares" else case["n_params"])
    if kind == "estimate":
        groups = 1 if case["strategy"] == "aggregate" else n * (n + 1) // 2 if case["quantity"] == "hessian" else n
        renders, io = groups * case["samples"], 8 * (n + n * n)
    elif kind == "newton":
        renders = case["instances"] * (case["n_grad"] + case["cg_iters"] * case["n_hvp"])
        io = 16 * n * case["instances"]
    elif kind == "optimise":
        renders = case["evals"] * case["instances"] * (case["n_grad"] + case["n_hvp"])
        io = 16 * n * case["instances"]
    else:
        renders, io = 3 * case["samples"] * case["requests"], 8 * 6 * case["requests"]
    channels = 1 if scene in ("disc", "squares") else 3
    flops = renders * _render_flops(scene, w, h, verts, tris, case.get("spp", 1), case.get("squares", 0))
    return dict(bytes=4 * w * h * channels + 12 * (verts + tris) + io, flops=flops)


# ---------------------------------------------------------------------------
# the method in 64 bits
# ---------------------------------------------------------------------------
M32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 (Salmon et al. 2011) on int64 tensors holding 32-bit words."""
    k0, k1 = seed & M32, (seed >> 32) & M32
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
        a, b = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((b >> 32) & M32) ^ c1 ^ k0, b & M32, ((a >> 32) & M32) ^ c3 ^ k1, a & M32
    return c0, c1, c2, c3


def _u01(x):
    return (x.to(F64) + 0.5) * 2.0 ** -32


def _u24(x):
    return (x >> 8).to(F64) * 2.0 ** -24 + 2.0 ** -25


def _lobe_t(c):
    """Inverse of the diagonal lobe's CDF: t^2 exp(-t^2) = 16 m^2 / e, tails t^2 >= 1, middle t^2 <= 1."""
    tail = (c < 0.25) | (c > 0.75)
    m = torch.where(tail, torch.minimum(c, 1.0 - c), (c - 0.5).abs()).clamp_min(1e-300)
    L = -2.0 * torch.log(4.0 * m)
    u = torch.sqrt(2.0 * L.clamp_min(0.0))
    y = torch.exp(-1.0 - L)
    up = torch.where(u < 2.0, 1.0 + u + u * u / 3.0, 1.0 + L + torch.log(1.0 + L))
    low = torch.where(u < 1.0, 1.0 - u + u * u / 3.0, y * (1.0 + y))
    s = torch.where(tail, up, low)
    for _ in range(30):   # Halley on log s - s + 1 + L = 0
        g, om = torch.log(s) - s + 1.0 + L, 1.0 - s
        sn = s - 2.0 * g * om * s / (2.0 * om * om + g)
        sn = torch.where(sn > 0.0, sn, 0.5 * s)
        wrong = torch.where(tail, sn < 1.0, sn > 1.0)
        s = torch.where((u > 1e-6) & torch.isfinite(sn), torch.where(wrong, 0.5 * (s + 1.0), sn), s)
    t = torch.sqrt(s)
    return torch.where(torch.where(tail, c < 0.25, c < 0.5), -t, t)


def _draw(n, sigma, pairs, seed, request, sub, lobe, comp=None, row=None, v=None):
    """[2 pairs][n] perturbations in 32 bits.  lobe 0: gradient, 1: Hessian; comp: one element (i, j) or None
    for the mixture of all; row: the row mixture of an element-wise HVP along v.  `request` and `sigma` may
    be tensors of one value a pair (several instances at once)."""
    k = torch.arange(pairs, dtype=torch.int64, device=DEV) if isinstance(pairs, int) else pairs
    c2 = (1 << 24) | sub
    zg = math.sqrt(2.0 / math.pi) / sigma
    zd, zo = 4.0 * math.exp(-0.5) / math.sqrt(2.0 * math.pi) / sigma ** 2, zg * zg
    w = _philox(k, torch.zeros_like(k), torch.zeros_like(k) + c2, torch.zeros_like(k) + request, seed)
    if row is not None:
        mass = torch.tensor(np.abs(v) * np.where(np.arange(n) == row, zd, zo), device=DEV)
        i = torch.full_like(k, row)
        j = torch.searchsorted(torch.cumsum(mass, 0), _u01(w[0]) * mass.sum(), right=True).clamp_max(n - 1)
    elif comp is not None:
        i, j = torch.full_like(k, comp[0]), torch.full_like(k, comp[1] if lobe else comp[0])
    elif lobe == 0:
        i = j = (w[0] * n) >> 32
    else:
        e = (w[0] * (n * n)) >> 32
        i, j = e // n, e % n
    g = torch.zeros((k.numel(), (n + 3) // 4 * 4), dtype=F64, device=DEV)
    for d in range(0, n, 4):
        r = _philox(k, torch.zeros_like(k) + 1 + d // 4, torch.zeros_like(k) + c2, torch.zeros_like(k) + request, seed)
        for h in range(2):
            rad, ph = torch.sqrt(-2.0 * torch.log(_u01(r[2 * h]))), 2.0 * math.pi * _u01(r[2 * h + 1])
            g[:, d + 2 * h], g[:, d + 2 * h + 1] = sigma * (rad * torch.cos(ph)), sigma * (rad * torch.sin(ph))
    g = g[:, :n]
    ua, ub = _u01(w[1]), _u01(w[2])
    ra, rb = sigma * torch.sqrt(-2.0 * torch.log(ua)), sigma * torch.sqrt(-2.0 * torch.log(ub))
    if lobe == 0:
        legs = [(ra, ra), (-ra, -ra)]
    else:
        tail = sigma * _lobe_t(torch.where(ua < 0.5, 0.5 * ua, 0.5 + 0.5 * ua))
        middle = sigma * _lobe_t(0.25 + 0.5 * ua)
        sg = torch.where((w[3] & 1) == 1, -1.0, 1.0)
        legs = [(torch.where(i == j, tail, sg * ra), torch.where(i == j, tail, sg * rb)),
                (torch.where(i == j, middle, sg * ra), torch.where(i == j, middle, -sg * rb))]
    out = []
    for vi, vj in legs:
        t = g.clone()
        t.scatter_(1, j[:, None], vj[:, None])
        t.scatter_(1, i[:, None], vi[:, None])
        out.append(t.to(torch.float32))
    return torch.stack(out, 1).reshape(-1, n)


def _inverse_density(t, sigma, lobe):
    """N(t) / q(t) of the mixture of all gradient or all (ordered) Hessian lobes, [..., n] -> [...]."""
    n = t.shape[-1]
    zg = math.sqrt(2.0 / math.pi) / sigma
    if lobe == 0:
        return 1.0 / (t.abs().sum(-1) / sigma ** 2 / zg / n)
    zd = 4.0 * math.exp(-0.5) / math.sqrt(2.0 * math.pi) / sigma ** 2
    off = t.abs().sum(-1) ** 2 - (t * t).sum(-1)
    return n * n / ((t * t - sigma ** 2).abs().sum(-1) / sigma ** 4 / zd + off / sigma ** 4 / (zg * zg))


def _estimate_exact(sc, target, quantity, strategy, theta, v, sigma, m, seed, request):
    """One estimate: draws, losses of all renders, weighted mean."""
    n = sc["n_params"]
    theta32 = torch.tensor(np.asarray(theta, np.float64), device=DEV).to(torch.float32)

    def losses(tau, sub):
        k = torch.arange(m // 2, device=DEV).repeat_interleave(2)
        return _losses(sc, target, theta32 + tau, seed, request, sub, k)

    if strategy == "aggregate":
        t32 = _draw(n, sigma, m // 2, seed, request, 0, 0 if quantity == "grad" else 1)
        f, t = losses(t32, 0), t32.to(F64)
        fw = f * _inverse_density(t, sigma, 0 if quantity == "grad" else 1) / m
        if quantity == "grad":
            return (fw[:, None] * t).sum(0) / sigma ** 2
        if quantity == "hessian":
            return (t.T * fw) @ t / sigma ** 4 - torch.eye(n, dtype=F64, device=DEV) * fw.sum() / sigma ** 2
        vv = torch.tensor(v, device=DEV)
        return (t.T @ (fw * (t @ vv))) / sigma ** 4 - vv * fw.sum() / sigma ** 2
    sign = torch.tensor([1.0, -1.0], dtype=F64, device=DEV).repeat(m // 2)
    zg = math.sqrt(2.0 / math.pi) / sigma
    zd = 4.0 * math.exp(-0.5) / math.sqrt(2.0 * math.pi) / sigma ** 2
    if quantity == "grad":
        return torch.stack([zg * (sign * losses(_draw(n, sigma, m // 2, seed, request, e, 0, (e, e)), e)).mean()
                            for e in range(n)])
    if quantity == "hessian":
        out = torch.zeros((n, n), dtype=F64, device=DEV)
        pairs = [(i, j) for i in range(n) for j in range(i, n)]
        for e, (i, j) in enumerate(pairs):
            out[i, j] = out[j, i] = (zd if i == j else zg * zg) * \
                (sign * losses(_draw(n, sigma, m // 2, seed, request, e, 1, (i, j)), e)).mean()
        return out
    rows = []
    for i in range(n):
        t32 = _draw(n, sigma, m // 2, seed, request, i, 1, row=i, v=v)
        t, av = t32.to(F64), torch.tensor(np.abs(v), device=DEV)
        c = t[:, i:i + 1] * t / sigma ** 4
        c[:, i] -= 1.0 / sigma ** 2
        z = torch.full((n,), zg * zg, dtype=F64, device=DEV)
        z[i] = zd
        weight = (c @ torch.tensor(v, device=DEV)) * (av * z).sum() / (c.abs() @ av)
        rows.append((weight * losses(t32, i)).mean())
    return torch.stack(rows)


def _losses(sc, target, p32, seed, request, sub, k):
    """Mean squared difference to the target of the renders at p32 [M][n] (perturbed parameters in 32 bits)."""
    npx = sc["width"] * sc["height"]
    many = {wl.SCENE_PTBOX: (1 << 21) // (npx * sc.get("spp", 1)), wl.SCENE_REVOLVE3D: (1 << 28) // npx}
    step = max(1, many.get(sc["kind"], (1 << 24) // npx))
    out = []
    for b in range(0, len(p32), step):
        req = request if isinstance(request, int) else request[b:b + step]
        img = _images(sc, p32[b:b + step], seed, req, sub, k[b:b + step], 2, sc.get("spp", 1))
        out.append((img - target).square_().flatten(1).mean(1))
    return torch.cat(out)


def _target(sc):
    p = torch.tensor(np.asarray(sc["theta_target"], np.float64), device=DEV).to(torch.float32)[None]
    zero = torch.zeros(1, dtype=torch.int64, device=DEV)
    if sc["kind"] != wl.SCENE_PTBOX:
        return _images(sc, p, 0, 0, 0, zero, 3, 1)
    return _images(sc, p, sc["seed"], 0, 0, zero, 3, sc["target_spp"])


def _images(sc, p32, seed, request, sub, k, tag, spp):
    p = p32.to(F64)
    w, h = sc["width"], sc["height"]
    x = torch.arange(w, dtype=F64, device=DEV) + 0.5
    y = (torch.arange(h, dtype=F64, device=DEV) + 0.5)[:, None]
    if sc["kind"] == wl.SCENE_DISC2D:
        r = float(sc["radius"])
        return ((x / w - p[:, 0, None, None]) ** 2 + (y / h - p[:, 1, None, None]) ** 2 < r * r).to(F64)
    if sc["kind"] == wl.SCENE_BOXES2D:
        s, out = float(sc["half_size"]), torch.zeros((len(p), h, w), dtype=torch.bool, device=DEV)
        for q in range(p.shape[1] // 2):
            out |= ((x / w - p[:, 2 * q, None, None]).abs() < s) & ((y / h - p[:, 2 * q + 1, None, None]).abs() < s)
        return out.to(F64)
    if sc["kind"] == wl.SCENE_TRIS2D:
        return _tris_images(sc, p, x, y)
    if sc["kind"] == wl.SCENE_REVOLVE3D:
        return _mesh_images(sc, p)
    return _ptbox_images(sc, p, seed, request, sub, k, tag, spp)


def _edges(ax, ay, bx, by, x, y):
    return (by - ay) * x + (ax - bx) * y + (ay * bx - ax * by)


def _tris_images(sc, p, x, y):
    """Painter's order, both windings; [M][H][W][3]."""
    raw = torch.tensor(np.asarray(sc["raw_params"], np.float64), device=DEV).repeat(len(p), 1)
    raw[:, torch.tensor(np.asarray(sc["param_index"], np.int64), device=DEV)] = p
    raw = raw.reshape(len(p), sc["n_tris"], 9, 1, 1)
    img = torch.zeros((len(p), sc["height"], sc["width"], 3), dtype=F64, device=DEV)
    for t in range(sc["n_tris"]):
        q = raw[:, t]
        ax, ay, bx, by, cx, cy = (q[:, c] * (sc["width"], sc["height"])[c % 2] for c in range(6))
        s = torch.sign(_edges(ax, ay, bx, by, cx, cy))
        inside = (s * _edges(bx, by, cx, cy, x, y) > 0) & (s * _edges(cx, cy, ax, ay, x, y) > 0) & \
            (s * _edges(ax, ay, bx, by, x, y) > 0)
        img = torch.where(inside[..., None], q[:, 6:9].reshape(-1, 1, 1, 3), img)
    return img


def _mesh_images(sc, p):
    """Perspective raster, back faces culled, largest 1/Z wins, flat Lambert shade; [M][H][W][3]."""
    w, h, m = sc["width"], sc["height"], len(p)
    vert = torch.tensor(np.asarray(sc["vertices"], np.float64), device=DEV)
    tri = torch.tensor(np.asarray(sc["triangles"], np.int64), device=DEV)
    ca, sa, cb, sb = torch.cos(p[:, 0]), torch.sin(p[:, 0]), torch.cos(p[:, 1]), torch.sin(p[:, 1])
    zero = torch.zeros_like(ca)
    rot = torch.stack([cb, zero, sb, sa * sb, ca, -sa * cb, -ca * sb, sa, ca * cb], 1).reshape(m, 3, 3)
    cam = torch.einsum("mrc,vc->mvr", rot, vert)
    z = float(sc["eye_dist"]) - cam[..., 2]
    sx, sy = float(sc["scale"]) * cam[..., 0] / z + 0.5 * w, -float(sc["scale"]) * cam[..., 1] / z + 0.5 * h
    nrm = torch.linalg.cross(vert[tri[:, 1]] - vert[tri[:, 0]], vert[tri[:, 2]] - vert[tri[:, 0]])
    nrm = nrm / nrm.norm(dim=1, keepdim=True).clamp_min(1e-300)
    light = torch.tensor(np.asarray(sc["light"], np.float64), device=DEV)
    shade = (torch.einsum("mrc,tc->mtr", rot, nrm) @ light).clamp_min(0.0)
    X, Y, W = sx[:, tri], sy[:, tri], 1.0 / z[:, tri]
    area = _edges(X[..., 0], Y[..., 0], X[..., 1], Y[..., 1], X[..., 2], Y[..., 2])
    lo_x, hi_x = torch.ceil(X.amin(2) - 0.5).clamp_min(0).long(), torch.floor(X.amax(2) - 0.5).clamp_max(w - 1).long()
    lo_y, hi_y = torch.ceil(Y.amin(2) - 0.5).clamp_min(0).long(), torch.floor(Y.amax(2) - 0.5).clamp_max(h - 1).long()
    seen = (area > 0) & (hi_x >= lo_x) & (hi_y >= lo_y) & (z[:, tri] > 0).all(2)
    wide = torch.where(seen, hi_x - lo_x + 1, 0).amax(0).tolist()
    high = torch.where(seen, hi_y - lo_y + 1, 0).amax(0).tolist()
    depth = torch.zeros(m * w * h, dtype=F64, device=DEV)
    img = torch.zeros(m * w * h, dtype=F64, device=DEV)
    for t in range(len(tri)):
        if not wide[t]:
            continue
        at = torch.nonzero(seen[:, t])[:, 0]
        c = lambda a: a[at, t, None, None]   # noqa: E731
        ix, iy = c(lo_x) + torch.arange(wide[t], device=DEV), c(lo_y) + torch.arange(high[t], device=DEV)[:, None]
        x, y = ix + 0.5, iy + 0.5
        (ax, bx, cx), (ay, by, cy), (wa, wb, wc) = ([a[at, t, q, None, None] for q in range(3)] for a in (X, Y, W))
        e0, e1, e2 = _edges(bx, by, cx, cy, x, y), _edges(cx, cy, ax, ay, x, y), _edges(ax, ay, bx, by, x, y)
        inv = (e0 * wa + e1 * wb + e2 * wc) / c(area)
        pos = at[:, None, None] * (w * h) + iy.clamp_max(h - 1) * w + ix.clamp_max(w - 1)
        hit = (e0 > 0) & (e1 > 0) & (e2 > 0) & (ix <= c(hi_x)) & (iy <= c(hi_y)) & (inv > depth[pos])
        pos = pos[hit]
        depth[pos] = inv[hit]
        img[pos] = c(shade).expand(hit.shape)[hit]
    albedo = torch.tensor(np.asarray(sc["albedo"], np.float64), device=DEV)
    return img.reshape(m, h, w, 1) * albedo


def _ptbox_images(sc, p, seed, request, sub, k, tag, spp):
    """Path tracer: next-event estimation, cosine-weighted continuation, fixed depth 3; [M][H W][3]."""
    w, h, m = sc["width"], sc["height"], len(p)
    if spp > 16 and m == 1:   # a target: in slices of its samples' pixels
        return torch.cat([_ptbox_paths(sc, p, seed, request, sub, k, tag, spp, b, min(w * h, b + 4096))
                          for b in range(0, w * h, 4096)], 1)
    return _ptbox_paths(sc, p, seed, request, sub, k, tag, spp, 0, w * h)


def _dot(a, b):
    return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]


def _ptbox_paths(sc, p, seed, request, sub, k, tag, spp, first, last):
    w, m, npx = sc["width"], len(p), last - first
    each = npx * spp
    idx = torch.arange(first * spp, last * spp, device=DEV).repeat(m)
    P = [p[:, c].repeat_interleave(each) for c in range(6)]
    kk = k.repeat_interleave(each)
    c2 = torch.zeros_like(idx) + ((tag << 24) | sub)
    req = torch.zeros_like(idx) + (request if isinstance(request, int) else request.repeat_interleave(each))
    half, depth = float(sc["light_half"]), int(sc.get("depth", 3))
    quads = [(int(a), *(float(c) for c in g)) for a, g in zip(sc["quad_axis"], sc["quad_geom"])]
    quads.append((1, P[1], P[0] - half, P[2] - half, P[0] + half, P[2] + half))
    centres = [[float(c) for c in s] for s in sc["sph_center"]]
    centres[0] = P[3:6]
    albedo = torch.tensor(np.concatenate([sc["quad_albedo"], np.zeros((1, 3)), sc["sph_albedo"]]).astype(np.float64), device=DEV)
    axis = torch.tensor([q[0] for q in quads] + [0, 0, 0], device=DEV)

    def closest(o, d):
        best, prim = torch.full_like(d[0], math.inf), torch.full_like(idx, -1)
        for q, (a, plane, lo_u, lo_v, hi_u, hi_v) in enumerate(quads):
            u, v = (1 if a == 0 else 0), (1 if a == 2 else 2)
            t = (plane - o[a]) / d[a]
            hu, hv = o[u] + t * d[u], o[v] + t * d[v]
            ok = (d[a] != 0) & (t > 0) & (hu >= lo_u) & (hu <= hi_u) & (hv >= lo_v) & (hv <= hi_v) & (t < best)
            best, prim = torch.where(ok, t, best), torch.where(ok, q, prim)
        for s in range(3):
            oc = [o[c] - centres[s][c] for c in range(3)]
            b = _dot(oc, d)
            disc = b * b - (_dot(oc, oc) - float(sc["sph_radius"][s]) ** 2)
            root = torch.sqrt(disc.clamp_min(0.0))
            t = torch.where(-b - root > 0, -b - root, root - b)
            ok = (disc >= 0) & (t > 0) & (t < best)
            best, prim = torch.where(ok, t, best), torch.where(ok, 13 + s, prim)
        return best, prim

    def words(block):
        return _philox(idx, (kk << 8) | block, c2, req, seed)

    px = idx // spp
    j = words(0)
    x, y = (px % w).to(F64) + _u24(j[0]), (px // w).to(F64) + _u24(j[1])
    d = [x * float(sc["pix_scale"]) - float(sc["tan_half"]), float(sc["tan_half"]) - y * float(sc["pix_scale"]),
         torch.full_like(x, -1.0)]
    inv = 1.0 / torch.sqrt(_dot(d, d))
    d = [c * inv for c in d]
    o = [torch.zeros_like(x), torch.zeros_like(x), torch.full_like(x, float(sc["cam_z"]))]
    emit = [float(c) for c in sc["light_emission"]]
    t, prim = closest(o, d)
    L = [torch.where((prim == 12) & (d[1] > 0), c, 0.0).to(F64) for c in emit]
    beta = [torch.ones_like(x) for _ in range(3)]
    area = (2.0 * half) ** 2
    for vertex in range(1, depth + 1):
        live = (prim >= 0) & (prim != 12)
        t = torch.where(live, t, 0.0)
        pos = [o[c] + t * d[c] for c in range(3)]
        ax = axis[prim.clamp_min(0)]
        n = [torch.where(ax == c, torch.where(d[c] > 0, -1.0, 1.0), 0.0).to(F64) for c in range(3)]
        for s in range(3):
            on = prim == 13 + s
            ns = [(pos[c] - centres[s][c]) / float(sc["sph_radius"][s]) for c in range(3)]
            flip = torch.where(_dot(ns, d) > 0, -1.0, 1.0)
            n = [torch.where(on, ns[c] * flip, n[c]) for c in range(3)]
        o2 = [pos[c] + 1e-4 * n[c] for c in range(3)]
        rho = albedo[prim.clamp_min(0)]
        r = words(vertex << 4)
        lp = [P[0] - half + _u24(r[0]) * 2 * half, P[1], P[2] - half + _u24(r[1]) * 2 * half]
        to = [lp[c] - o2[c] for c in range(3)]
        dist2 = _dot(to, to)
        om = [c / torch.sqrt(dist2) for c in to]
        cosx = _dot(n, om)
        lit = live & (cosx > 0) & (om[1] > 0) & (closest(o2, om)[1] == 12)
        geo = torch.where(lit, cosx * om[1] / dist2 * area / math.pi, 0.0)
        L = [L[c] + beta[c] * rho[:, c] * emit[c] * geo for c in range(3)]
        if vertex == depth:
            break
        tries = [(r[2], r[3])]
        for block in (1, 2, 3):
            q = words((vertex << 4) | block)
            tries += [(q[0], q[1]), (q[2], q[3])]
        a, b, found = torch.zeros_like(x), torch.zeros_like(x), torch.zeros_like(live)
        for qa, qb in tries:
            ta, tb = _u24(qa) * 2 - 1, _u24(qb) * 2 - 1
            take = ~found & (ta * ta + tb * tb < 1)
            a, b, found = torch.where(take, ta, a), torch.where(take, tb, b), found | take
        cz = torch.sqrt((1 - (a * a + b * b)).clamp_min(0.0))
        sg = torch.where(n[2] >= 0, 1.0, -1.0)   # basis around n: Duff et al. 2017
        aa = -1.0 / (sg + n[2])
        bb = n[0] * n[1] * aa
        t1 = [1 + sg * n[0] * n[0] * aa, sg * bb, -sg * n[0]]
        t2 = [bb, sg + n[1] * n[1] * aa, -n[1]]
        beta = [beta[c] * rho[:, c] for c in range(3)]
        o, d = o2, [cz * n[c] + b * t2[c] + a * t1[c] for c in range(3)]
        t, nxt = closest(o, d)
        prim = torch.where(live, nxt, -1)
    return torch.stack(L, 1).reshape(m, npx, spp, 3).mean(2)


def _optimiser_options(case, seed):
    return dict(sigma_start=0.1, sigma_end=0.01, anneal_iters=30, n_grad=case["n_grad"], n_hvp=case["n_hvp"], ls_iters=2,
                ls_tol=1e-3, recompute=1, residual_mode=0, trust_radius=0.02, lambda_rel=0.0, seed=seed, request_base=0,
                use_graph=1)


def _instance_sums(sc, target, theta, sigma, m, seed, sub, lobe):
    """Perturbations [B][m][n] of B instances (request = instance) and their losses times N/q / m, [B][m];
    sigma: [B]."""
    B, n = theta.shape
    t32 = torch.stack([_draw(n, float(sigma[b]), m // 2, seed, b, sub, lobe) for b in range(B)])
    p = (torch.tensor(theta, device=DEV).to(torch.float32)[:, None] + t32).reshape(B * m, n)
    k = torch.arange(m // 2, device=DEV).repeat_interleave(2).repeat(B)
    f = _losses(sc, target, p, seed, torch.arange(B, device=DEV).repeat_interleave(m), sub, k).reshape(B, m)
    t = t32.to(F64)
    return t, torch.stack([f[b] * _inverse_density(t[b], float(sigma[b]), lobe) / m for b in range(B)])


def _newton_exact(case, seed):
    sc = _scene_dict(case, seed)
    target, theta, sigma = _target(sc), np.array(sc["theta_init"]), sc["sigma"]
    B = case["instances"]
    sig = np.full(B, sigma)
    t, fw = _instance_sums(sc, target, theta, sig, case["n_grad"], seed, 0, 0)
    g = ((fw[..., None] * t).sum(1) / sigma ** 2).cpu().numpy()
    products = [_instance_sums(sc, target, theta, sig, case["n_hvp"], seed, 1 + i, 1) for i in range(case["cg_iters"])]
    steps, norms = np.zeros_like(theta), np.linalg.norm(g, axis=1)
    for b in range(B):
        d, r = np.zeros(theta.shape[1]), -g[b]
        p, rr = r.copy(), r @ r
        for i, (t, fw) in enumerate(products):
            tb, fb = t[b].cpu().numpy(), fw[b].cpu().numpy()
            hp = tb.T @ (fb * (tb @ p)) / sigma ** 4 - p * fb.sum() / sigma ** 2 + 1e-3 * norms[b] * p
            php, pn = p @ hp, np.linalg.norm(p)
            if not php > 0 or pn == 0:
                if i == 0 and pn > 0:
                    d = p * (0.05 / pn)
                break
            alpha = min(rr / php, 0.05 / pn)
            d, r = d + alpha * p, r - alpha * hp
            new = r @ r
            if new == 0:
                break
            p, rr = r + new / rr * p, new
        steps[b] = d
    return dict(theta=theta + steps, grad_norm=norms, step_norm=np.linalg.norm(steps, axis=1), iters=None)


def _optimise_exact(case, seed):
    sc, theta = _optimise_inputs(case, seed)
    target, o, B = _target(sc), _optimiser_options(case, seed), case["instances"]
    d, it, ls = np.zeros_like(theta), np.zeros(B, int), np.zeros(B, int)
    norms, alphas = [], []
    for e in range(case["evals"]):
        sig = o["sigma_start"] + (o["sigma_end"] - o["sigma_start"]) * np.minimum(it, 29) / 29
        s2 = torch.tensor(sig ** 2, device=DEV)[:, None]
        t, fw = _instance_sums(sc, target, theta, sig, o["n_grad"], seed, 64 * e, 0)
        g = ((fw[..., None] * t).sum(1) / s2).cpu().numpy()
        t, fw = _instance_sums(sc, target, theta, sig, o["n_hvp"], seed, 64 * e + 1, 1)
        d = np.where(ls[:, None] == 0, -g, d)   # recompute = 1: every outer iteration restarts along -g
        dd = torch.tensor(d, device=DEV)
        q = torch.einsum("bmn,bm->bn", t, fw * torch.einsum("bmn,bn->bm", t, dd)) / s2 ** 2 - dd * fw.sum(1)[:, None] / s2
        gd, dhd, dn = (g * d).sum(1), (d * q.cpu().numpy()).sum(1), np.linalg.norm(d, axis=1)
        cap = o["trust_radius"] / np.where(dn > 0, dn, 1)
        alpha = np.where(dhd > 0, -gd / np.where(dhd > 0, dhd, 1), np.where(gd < 0, cap, np.where(gd > 0, -cap, 0)))
        alpha = np.where(dn > 0, np.clip(alpha, -cap, cap), 0.0)
        theta = theta + alpha[:, None] * d
        norms.append(np.linalg.norm(g, axis=1))
        alphas.append(alpha)
        done = (ls + 1 >= o["ls_iters"]) | (np.abs(alpha) * dn <= o["ls_tol"])
        it, ls = it + done, np.where(done, 0, ls + 1)
    return dict(theta=theta, grad_norm=np.concatenate(norms), alpha=np.concatenate(alphas))


def exact(case, seed):
    kind = case["kind"]
    if kind == "newton":
        return _newton_exact(case, seed)
    if kind == "optimise":
        return _optimise_exact(case, seed)
    if kind == "queue":
        sc, thetas, seeds = _queue_inputs(case, seed)
        target = _target(sc)
        return torch.stack([_estimate_exact(sc, target, "hessian", "elementwise", th, None, sc["sigma"], case["samples"],
                                            int(s), i) for i, (th, s) in enumerate(zip(thetas, seeds))]).cpu()
    if kind == "serve":
        scenes, reqs = _serve_inputs(case, seed)
        targets = {k: _target(scenes[k]) for k in {r["scene"] for r in reqs}}
        names, how = {v: k for k, v in QUANTITY.items()}, {v: k for k, v in STRATEGY.items()}
        return [_estimate_exact(scenes[r["scene"]], targets[r["scene"]], names[r["quantity"]], how[r["strategy"]],
                                r["theta"], r["v"], r["sigma"], r["M"], r["seed"], r["request"]).cpu() for r in reqs]
    sc = _scene_dict(case, seed)
    v = _direction(sc, seed) if case["quantity"] == "hvp" else None
    return _estimate_exact(sc, _target(sc), case["quantity"], case["strategy"], sc["theta_query"], v, sc["sigma"],
                           case["samples"], seed, 0).cpu()
