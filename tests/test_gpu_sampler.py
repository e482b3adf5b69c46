"""The sampler's blocks of pairs and the estimator sums at the sizes where their
launches change: dims per warp, ragged last blocks, many weights per row, rows
per chunk."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2412_03489_gb300 import build as hb
from paper_2412_03489_gb300 import hr
from paper_2412_03489_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

hb.build()

Q = {"grad": hr.HR_GRAD, "hessian": hr.HR_HESSIAN, "hvp": hr.HR_HVP}
S = {"elementwise": hr.HR_ELEMENTWISE, "aggregate": hr.HR_AGGREGATE, "plain": hr.HR_PLAIN}


def scene(n):
    g = np.random.default_rng(n)
    return wl.quadratic_scene(A=g.normal(size=(n, n)), b=g.normal(size=n), theta=g.normal(size=n), sigma=0.1)


def run(sc, quantity, strategy, M, seed=3, request=4, sub=5):
    v = np.random.default_rng(7).normal(size=sc["n_params"])
    s = hr.Scene(sc)
    out, d = s.estimate(Q[quantity], sc["theta_query"], sc["sigma"], M, S[strategy], seed, request, sub,
                        v=v if quantity == "hvp" else None, debug=True)
    s.close()
    return out, d, v


@pytest.mark.parametrize("n", [1, 2, 3, 15, 16, 33, 64])
@pytest.mark.parametrize("quantity", ["grad", "hessian", "hvp"])
@pytest.mark.parametrize("strategy", ["elementwise", "aggregate", "plain"])
def test_draws_and_weights_against_the_oracle(n, quantity, strategy):
    if strategy == "elementwise" and quantity == "hessian" and n > 3:
        pytest.skip("one group per element: covered by the small n")
    sc = scene(n)
    M = 2 * 37 if strategy != "elementwise" else 2 * 5
    _, d, v = run(sc, quantity, strategy, M)
    r = O.FunctionRenderer(lambda P: np.zeros(len(P)), n)
    ref = O.estimate(r, quantity, sc["theta_query"], sc["sigma"], M, strategy, 3, 4, sub=5,
                     v=v if quantity == "hvp" else None)
    assert np.array_equal(d["tau"], ref.tau)
    # both sides round an FP64 weight to FP32: a unit in the last place
    assert np.allclose(d["w"], ref.w.astype(np.float32), rtol=2e-7, atol=2e-7 * np.abs(ref.w).max())


@pytest.mark.parametrize("n,M", [(16, 600), (47, 260), (64, 130)])
def test_off_diagonal_weights_are_rounded_as_in_fp64(n, M):
    """The mixture's off-diagonal weights, formed without FP64 where that is
    certain, against the FP64 products rounded once.  The density S may differ from
    this restatement's in its last bits (relative 1e-14), which moves a
    weight across a rounding boundary with a probability of about 1e-14 / 2^-25 =
    3e-7: fewer than one is expected among the 280,000 of a case."""
    sc = scene(n)
    _, d, _ = run(sc, "hessian", "aggregate", M)
    t, s2 = d["tau"].astype(np.float64), sc["sigma"] ** 2
    zg = np.sqrt(2 / np.pi) / sc["sigma"]
    zd = 4 * np.exp(-0.5) / (np.sqrt(2 * np.pi) * s2)
    is4 = (1 / s2) * (1 / s2)
    sa, sq = np.abs(t).sum(1), (t * t).sum(1)
    dens = (np.abs(t * t - s2).sum(1) * is4 / zd + (sa * sa - sq) * is4 / zg ** 2) / n ** 2
    i, j = np.triu_indices(n)
    off = i != j
    want = (t[:, i] * t[:, j] * is4 / dens[:, None])[:, off].astype(np.float32)
    got = d["w"][:, off]
    assert np.count_nonzero(got != want) <= 5
    assert np.all(np.abs(got - want) <= np.spacing(np.abs(want)))


def sums(w, f, elementwise, M):
    """256 Kahan FP32 chunks per element and the FP64 tree (t, t + o), o = 128 .. 1."""
    E = w.shape[1]
    chunk = (M + 255) // 256
    out = np.zeros(E)
    for e in range(E):
        x = np.zeros(256 * chunk, np.float32)
        x[:M] = (w[e * M:(e + 1) * M, e] * f[e * M:(e + 1) * M]) if elementwise else w[:, e] * f
        x = x.reshape(256, chunk)
        s, c = np.zeros(256, np.float32), np.zeros(256, np.float32)
        for k in range(chunk):
            live = np.arange(256) * chunk + k < M
            y = x[:, k] - c
            t = s + y
            c = np.where(live, (t - s) - y, c)
            s = np.where(live, t, s)
        v = s.astype(np.float64) - c.astype(np.float64)
        for o in (128, 64, 32, 16, 8, 4, 2, 1):
            v = v[:o] + v[o:2 * o]
        out[e] = v[0] * (1.0 / M)
    return out


@pytest.mark.parametrize("n,quantity,strategy,M", [
    (2, "hessian", "aggregate", 2), (2, "hessian", "aggregate", 1024), (2, "hessian", "aggregate", 1026),
    (2, "hessian", "elementwise", 4098), (3, "grad", "aggregate", 8190), (2, "hvp", "plain", 16386),
    (10, "hessian", "aggregate", 1300), (45, "hessian", "aggregate", 258), (64, "hessian", "aggregate", 1100),
    (64, "grad", "aggregate", 1030),
])
def test_sums_keep_their_order(n, quantity, strategy, M):
    out, d, _ = run(scene(n), quantity, strategy, M)
    flat = out[np.triu_indices(n)] if quantity == "hessian" else out
    assert np.array_equal(flat, sums(d["w"], d["losses"], strategy == "elementwise", M))


@pytest.mark.parametrize("quantity,strategy", [("hessian", "elementwise"), ("grad", "aggregate"), ("hessian", "plain")])
def test_many_draws_equal_the_oracles(quantity, strategy):
    """Every draw of 8,192 perturbations per group: the sampler's own logarithm and
    the C library's differ by a unit in the last place of FP64 at most, which moves a
    value across an FP32 rounding boundary with a probability of about 2^-28: fewer
    than one in a thousand runs of the 50,000 values."""
    sc = scene(2)
    _, d, _ = run(sc, quantity, strategy, 8192)
    ref = O.estimate(O.FunctionRenderer(lambda P: np.zeros(len(P)), 2), quantity, sc["theta_query"], sc["sigma"], 8192,
                     strategy, 3, 4, sub=5)
    assert np.array_equal(d["tau"], ref.tau)


@pytest.mark.parametrize("n", [2, 16, 33])
@pytest.mark.parametrize("sigma", [1e-15, 1e-6, 1e9, 2e11, 3e11, 1e12, 1e18])
def test_weights_at_extreme_bandwidths(n, sigma):
    """Aggregate Hessian weights are of the order of 1 / sigma^2, a normal float here, although
    sigma^-4 is not one for the larger bandwidths (or for the smallest)."""
    sc = dict(scene(n), sigma=sigma)
    M = 2 * 21
    _, d, _ = run(sc, "hessian", "aggregate", M)
    ref = O.estimate(O.FunctionRenderer(lambda P: np.zeros(len(P)), n), "hessian", sc["theta_query"], sigma, M,
                     "aggregate", 3, 4, sub=5)
    assert np.array_equal(d["tau"], ref.tau)
    assert np.allclose(d["w"], ref.w.astype(np.float32), rtol=2e-7, atol=2e-7 * np.abs(ref.w).max())


@pytest.mark.parametrize("n", [1, 2, 4, 5, 6, 13, 33])
def test_large_launches_equal_the_other_shapes(n):
    """Launches large enough that a block takes 32 pairs (an odd number of dim pairs), with a
    ragged last block: the bits of the shapes with 8 and 64 pairs a block."""
    sc = scene(n)
    s, M = hr.Scene(sc), 2 * (256 * torch.cuda.get_device_properties(0).multi_processor_count + 37)
    v = np.random.default_rng(7).normal(size=n)
    outs = {}
    for legs in (32, 16, 128):
        hr.hr_set_tuning(s.handle, 0, legs)
        outs[legs] = [s.estimate(q, sc["theta_query"], sc["sigma"], M, st, 3, 4, v=v if q == hr.HR_HVP else None)
                      for q in (hr.HR_GRAD, hr.HR_HVP) for st in (hr.HR_AGGREGATE, hr.HR_PLAIN)]
    s.close()
    assert all(np.array_equal(a, b) for legs in (16, 128) for a, b in zip(outs[32], outs[legs]))
