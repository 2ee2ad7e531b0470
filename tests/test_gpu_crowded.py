"""Problems whose obstacles crowd the robot's way (2-D, few of them static, a large
share of their box filled) run the chunked kernel, everything else that the
point-owner kernel covers runs that one: both sides of each line of the rule against
the FP64 oracle, without trial launches, in the projection of one problem, of a batch
and in the serving loop."""
import math

import numpy as np
import pytest

from gpu_common import TOL_FP32, rel_err, scale_of
from paper_2309_08235_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    from paper_2309_08235_gb300 import build, priest

    build.build()
    return priest


def crowd(p):
    """Share of the centres' box, grown by the mean radius, that the discs fill."""
    c, r = np.asarray(p["center"]), np.asarray(p["semi"]).max(1).mean()
    return len(c) * math.pi * r * r / np.prod(c.max(0) - c.min(0) + 2 * r)


def traffic(n, share, dims=2, vmax=1.0, static=0, mask=7, seed=7, n_p=60):
    """n discs (3-D: balls of the same radius) that fill `share` of a 5 x 3 m box on the way
    (0, 0) -> (8, 0) in 4.8 s (straight line: 1.7 m/s); all but `static` move."""
    rng = np.random.default_rng(seed)
    r = 0.1
    for _ in range(60):  # share = n pi r^2 / ((5 + 2 r) (3 + 2 r))
        r = math.sqrt(share * (5 + 2 * r) * (3 + 2 * r) / (n * math.pi))
    c = np.stack([rng.uniform(2, 7, n), rng.uniform(-1.5, 1.5, n)] + [rng.uniform(-1, 1, n)] * (dims - 2), 1)
    c[0, :2], c[1, :2] = (2.0, -1.5), (7.0, 1.5)
    v = np.zeros((n, dims))
    v[static:, 0] = -0.1
    p = W.problem(dims, n_p, 0.08 * n_p, np.zeros(dims), np.eye(dims)[0] * 8.0, c, v, np.full((n, 2), r), vmax, 1.0,
                  seed=seed)
    p["bc_final_mask"] = mask
    return p


# name: problem, samples, chunked?
CASES = {
    "below": (lambda: traffic(20, 0.24), 300, False),
    "above": (lambda: traffic(20, 0.26), 300, True),
    "few": (lambda: traffic(11, 0.6), 300, False),
    "many_samples": (lambda: traffic(20, 0.9), 1400, False),
    "many_samples_full": (lambda: traffic(20, 1.1), 1400, True),
    "fast": (lambda: traffic(40, 1.5, vmax=3.0), 620, False),
    "fast_full": (lambda: traffic(40, 2.1, vmax=3.0), 620, True),
    "fast_few": (lambda: traffic(20, 1.17, vmax=3.0), 450, False),
    "fast_few_full": (lambda: traffic(20, 1.23, vmax=3.0), 450, True),
    "fast_few_seven": (lambda: traffic(20, 1.17, vmax=3.0, mask=1), 140, False),
    "fast_few_seven_full": (lambda: traffic(20, 1.23, vmax=3.0, mask=1), 140, True),
    "static": (lambda: traffic(40, 1.5, static=16), 300, False),
    "seven": (lambda: traffic(20, 0.9, mask=1), 300, False),
    "seven_full": (lambda: traffic(20, 1.1, mask=1), 300, True),
    "three_d": (lambda: traffic(40, 2.5, dims=3), 300, False),
    "too_large": (lambda: traffic(2048, 3.0, n_p=512), 6, False),  # beyond the chunked kernel's tables
}


@pytest.mark.parametrize("name", list(CASES))
def test_route_and_parity(P, oracle, name):
    make, n, chunked = CASES[name]
    p = make()
    K = 12
    xi = oracle.default_mean(p) + 1.0 * W.normals(len(name), (n, p["dims"] * 11))
    with P.Context(p, {"proj_iters": K}, precision=P.PRIEST_FP32) as ctx:
        before = ctx.launches()
        first = ctx.project(p, xi)
        mid = ctx.launches()
        xb, _, r, c1 = ctx.project(p, xi)
        assert mid - before == ctx.launches() - mid  # no trials on the first call
        assert P.priest_last_kernel(ctx.h) == (0 if chunked else 1)
    for a, b in zip(first, (xb, None, r, c1)):
        if b is not None:
            np.testing.assert_array_equal(a, b)
    idx = np.r_[0:n:max(1, n // 12), n - 1]
    xb_o, _ = oracle.project(p, xi[idx], K)
    r_o, c1_o = oracle.residual_cost(p, xb_o)
    assert rel_err(xb[idx], xb_o, scale_of(p)) < TOL_FP32
    assert rel_err(r[idx], r_o, 1.0) < TOL_FP32
    assert rel_err(c1[idx], c1_o, max(1.0, np.abs(c1_o).max())) < TOL_FP32
    assert np.count_nonzero(r_o > 1e-6) > 0


def plan_batch(P, probs, calls):
    """The batched solves, through one context's host buffers, of the lists of problems
    probs[k], k in calls: (kernel kind, results) of each."""
    cem = W.cem_settings(256, 10, 2)
    n = len(probs[0])
    z = [W.normals(50 + i, (2, 256, 22)) for i in range(n)]
    out = []
    with P.Context(probs[0][0], cem, precision=P.PRIEST_FP32) as ctx:
        for k in calls:
            structs, keep = zip(*[P.make_problem(p, cem, per_problem_shape=True) for p in probs[k]])
            res = (P.priest_result * n)()
            P.priest_plan_batch_host(ctx.h, list(structs), z, res)
            out.append((P.priest_last_kernel(ctx.h), [P.result_dict(r) for r in res]))
    return out


def test_batch_crosses_the_line(P):
    """A resident batch whose obstacles close in and disperse again between calls of one
    layout: each call's results are those of a context of its own."""
    probs = [[traffic(20, s, seed=60 + i) for i in range(3)] for s in (0.2, 1.2)]
    there_and_back = plan_batch(P, probs, (0, 1, 0, 1))
    assert [kind for kind, _ in there_and_back] == [1, 0, 1, 0]
    for k, (_, got) in enumerate(there_and_back):
        (_, want), = plan_batch(P, probs, (k % 2,))
        for a, b in zip(got, want):
            assert a["status"] == 0
            np.testing.assert_array_equal(a["best"], b["best"])
            np.testing.assert_array_equal(a["mu"], b["mu"])
            assert a["c_aug"] == b["c_aug"]


def test_mixed_batch_keeps_the_lists(P):
    probs = [[traffic(20, s, seed=60 + i) for i, s in enumerate((0.2, 1.2, 1.2))]]
    assert plan_batch(P, probs, (0,))[0][0] == 1


def test_served_crowded_request(P, oracle):
    """One CEM iteration: the least c_aug among the ConstraintEliteSet is the oracle's."""
    p = traffic(20, 1.2, seed=71)
    p["seed"] = 9
    cem = W.cem_settings(128, 12, 1)
    with P.Context(p, cem, precision=P.PRIEST_FP32) as ctx:
        got = ctx.wait(ctx.submit(p, cem))
    z = oracle.rng_normal(p["seed"], 128 * 22).reshape(1, 128, 22)
    want = oracle.plan(p, cem, z=z)
    assert got["status"] == 0
    assert abs(got["c_aug"] - want["c_aug"]) < TOL_FP32 * max(1.0, want["c_aug"])
