"""The set-up kernel's parts (step a0): the first sampling factor of the default
covariance, written without an elimination, equals the factor of the same
covariance given explicitly (every off-diagonal step of that elimination is
zero), and the basis / inverse part holds at the ends of its thread splits (one
time stamp per thread, Gram sums in slices) against the oracle."""
import numpy as np
import pytest

from gpu_common import TOL_FP32, TOL_FP64, rel_err, samples, scale_of, scene
from paper_2309_08235_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    from paper_2309_08235_gb300 import build, priest

    build.build()
    return priest


@pytest.mark.parametrize("dims", [2, 3])
def test_default_covariance_equals_the_same_one_given(P, oracle, dims):
    p = scene(dims=dims, n_obs=6, n_p=20)
    cem = W.cem_settings(32, 5, 2, dims=dims)
    cem["init_std"] = 0.75
    D = dims * 11
    z = W.normals(5, (2, 32, D))
    with P.Context(p, cem, precision=P.PRIEST_FP64_CHECK) as ctx:
        a = ctx.plan(p, z=z)
        b = ctx.plan(p, z=z, cov0=0.75 ** 2 * np.eye(D))
    for k in ("best", "mu", "r", "c_aug", "best_index"):
        assert np.array_equal(a[k], b[k]), k


# fewer stamps than Gram slices, one more than a warp, the largest (FP32: the
# FP64 projection's tables of that many stamps exceed one CTA)
@pytest.mark.parametrize("n_p,mask", [(2, 7), (7, 1), (9, 7), (33, 1), (511, 7), (512, 1)])
def test_basis_part_at_its_split_edges(P, oracle, n_p, mask):
    p = scene(n_obs=3, n_dyn=1, n_p=n_p, mask=mask)
    xi = samples(oracle, p, 3, std=0.5)
    cem = W.cem_settings(16, 3, 1)
    with P.Context(p, cem, precision=P.PRIEST_FP32 if n_p > 400 else P.PRIEST_FP64_CHECK) as ctx:
        xb, lam, r, c1 = ctx.project(p, xi, lam=np.zeros_like(xi))
    xb_o, lam_o = oracle.project(p, xi, 3)
    tol = TOL_FP32 if n_p > 400 else TOL_FP64
    assert rel_err(xb, xb_o, scale_of(p)) < tol
    assert rel_err(lam, lam_o, scale_of(p)) < tol
