"""The FP32 point-owner projection at the edges of its layouts: teams of four
and of two warps per sample, one warp, and two samples per warp (chosen by the
samples an SM holds), each at the time-stamp counts where a stride, a block of
two stamps per lane or the sample's lists end, with more active pairs than a list
holds, without obstacles, and with warm multipliers (the fixed columns' sums).
Every output is bitwise the one of screening every pair in every iteration, and
matches the FP64 oracle."""
import os

import numpy as np
import pytest

from gpu_common import TOL_FP32, rel_err, samples, scale_of, scene

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    from paper_2309_08235_gb300 import build, priest

    build.build()
    return priest


def sm_count():
    import torch

    return torch.cuda.get_device_properties(0).multi_processor_count


# samples per SM: 4 warps a sample up to two, 2 warps up to eight (3-D, seven
# columns), one warp, and two samples a warp beyond sixteen (2-D, five columns)
PER_SM = {"four": 1, "four_twice": 2, "mid": 5, "single": 12, "pair": 18}


def project(P, p, xi, K, lam0, lists):
    old = os.environ.get("PRIEST_NEIGHBOUR_LISTS")
    os.environ["PRIEST_NEIGHBOUR_LISTS"] = lists
    try:
        with P.Context(p, {"proj_iters": K}, precision=P.PRIEST_FP32, autotune=0) as ctx:
            out = ctx.project(p, xi, lam=lam0)
            assert P.priest_last_kernel(ctx.h) == 1
    finally:
        if old is None:
            os.environ.pop("PRIEST_NEIGHBOUR_LISTS")
        else:
            os.environ["PRIEST_NEIGHBOUR_LISTS"] = old
    return out


@pytest.mark.parametrize("n_p", [2, 31, 33, 64, 65, 256, 257, 512])
@pytest.mark.parametrize("form", list(PER_SM))
@pytest.mark.parametrize("dims,mask", [(2, 7), (3, 7), (2, 1)])
def test_layout_edges(P, oracle, dims, mask, form, n_p):
    n = PER_SM[form] * sm_count() - 3
    warm = n_p in (33, 65, 512)
    p = scene(dims=dims, n_obs=24, n_dyn=3, n_p=n_p, mask=mask, bounds=mask == 1, seed=n_p)
    check(P, oracle, p, n, warm, 8)


@pytest.mark.parametrize("dims,mask", [(2, 7), (3, 7), (2, 1)])
@pytest.mark.parametrize("form", list(PER_SM))
@pytest.mark.parametrize("kind", ["none", "pile"])
def test_empty_and_overflowing_lists(P, oracle, kind, form, dims, mask):
    n = PER_SM[form] * sm_count() - 3
    if kind == "none":
        p = scene(dims=dims, n_obs=1, n_dyn=0, n_p=50, mask=mask)
        p = dict(p, center=np.zeros((0, dims)), semi=np.zeros((0, 2)), vel=np.zeros((0, dims)), n_obs=0)
    else:  # every time stamp inside several obstacles: thousands of active pairs a sample
        p = scene(dims=dims, n_obs=40, n_dyn=5, n_p=70, mask=mask, radius=(3.0, 5.0))
    check(P, oracle, p, n, kind == "pile", 5)


def check(P, oracle, p, n, warm, K):
    xi = samples(oracle, p, n, seed=n % 97)
    lam0 = np.random.default_rng(4).normal(0.0, 0.1, xi.shape) if warm else None
    got = project(P, p, xi, K, lam0, "1")
    every = project(P, p, xi, K, lam0, "0")
    for a, b in zip(got, every):
        if a is not None:
            np.testing.assert_array_equal(a, b)
    xb, lam, r, c1 = got
    idx = np.r_[0:n:max(1, n // 9), n - 1]
    xb_o, lam_o = oracle.project(p, xi[idx], K, lam=None if lam0 is None else lam0[idx])
    r_o, c1_o = oracle.residual_cost(p, xb_o)
    assert rel_err(xb[idx], xb_o, scale_of(p)) < TOL_FP32
    if warm:
        assert rel_err(lam[idx], lam_o, 1.0) < TOL_FP32
    assert rel_err(r[idx], r_o, 1.0) < TOL_FP32
    assert rel_err(c1[idx], c1_o, max(1.0, np.abs(c1_o).max())) < TOL_FP32
