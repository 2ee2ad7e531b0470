"""The selection kernel (Alg. 1, ConstraintEliteSet and EliteSet) against a sort
of the same keys: the elites are the n_elite least (c_1 + r, index) among the
n_proj least (r, index), in that order, at the edges of its search (one element,
a warp, more elements than threads, sets of everything), with both final sorts
(ranks by counting up to 256 elites, bitonic beyond) and with exact ties: samples
without any residual, and repeated samples, which only their index tells apart."""
import numpy as np
import pytest

from gpu_common import TOL_FP64, rel_err, scale_of, scene
from paper_2309_08235_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    from paper_2309_08235_gb300 import build, priest

    build.build()
    return priest


@pytest.mark.parametrize("N,n_proj,n_elite", [(1, 1, 1), (2, 1, 1), (32, 32, 32), (33, 20, 20), (110, 80, 20), (129, 40, 1),
                                              (1000, 727, 100), (1024, 1024, 256), (1025, 700, 257), (2500, 1300, 300),
                                              (8192, 5000, 1024)])
@pytest.mark.parametrize("ties", ["none", "zero_r", "repeated", "all_equal"])
def test_elites_are_the_sorted_prefix(P, N, n_proj, n_elite, ties):
    far = ties == "zero_r"
    p = (W.problem(2, 20, 10.0, [0, 0], [5, 5], [[100, 100]], None, [[0.5, 0.5]], vmax=1e3, amax=1e3) if far
         else scene(n_obs=8, n_dyn=1, n_p=20))
    cem = W.cem_settings(N, 2, 1, n_proj=n_proj, n_elite=n_elite, dims=2)
    z = W.normals(9, (1, N, 22))
    if ties == "repeated":
        z[0] = z[0][np.arange(N) % max(1, N // 40)]
    elif ties == "all_equal":
        z[0] = z[0][:1]
    with P.Context(p, cem, precision=P.PRIEST_FP32, autotune=0) as ctx:
        ctx.plan(p, z=z)
        el, r, c1 = P.priest_read_elites(ctx.h, None, n_elite, N)
    r, c1, i = np.asarray(r), np.asarray(c1), np.arange(N)
    if far:
        assert not r.any()
    first = np.lexsort((i, r))[:n_proj]
    want = first[np.lexsort((first, (c1 + r)[first]))][:n_elite]
    np.testing.assert_array_equal(np.asarray(el), want)


@pytest.mark.parametrize("N,n_elite", [(8192, 1024), (8161, 5), (300, 257)])
def test_batched_selection_equals_the_single_one(P, N, n_elite):
    """The batched launch's 256 threads hold up to 32 samples each; FP64 mode,
    where both launches project to the same bits up to rounding."""
    p = scene(n_obs=4, n_dyn=1, n_p=20)
    cem = W.cem_settings(N, 2, 2, n_proj=max(n_elite, N // 2), n_elite=n_elite, dims=2)
    z = W.normals(12, (2, N, 22))
    with P.Context(p, cem, precision=P.PRIEST_FP64_CHECK, autotune=0) as ctx:
        one = ctx.plan(p, z=z)
        struct, keep = P.make_problem(p, cem, per_problem_shape=True)
        res = (P.priest_result * 1)()
        P.priest_plan_batch_host(ctx.h, [struct], [z], res)
        both = P.result_dict(res[0])
    assert both["best_index"] == one["best_index"]
    assert rel_err(both["best"], one["best"], scale_of(p)) < TOL_FP64
    assert rel_err(both["mu"], one["mu"], scale_of(p)) < TOL_FP64
