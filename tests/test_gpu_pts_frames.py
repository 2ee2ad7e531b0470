"""The FP32 point-owner projection far from the frame's origin, with outlying
coefficients and with a margin below FP32's resolution: where coefficients round
coarsely the node test's own rounding can exceed its threshold, and an iteration
must still be done at most twice, with bitwise the results of screening every pair
in every iteration.  Teams of four and of two warps per sample, one warp, and two
samples per warp."""
import os

import numpy as np
import pytest

from gpu_common import TOL_FP32, samples, scale_of, scene
from test_gpu_pts_edges import P, PER_SM, project, sm_count  # noqa: F401

pytestmark = pytest.mark.gpu

K = 8
U = 2.0 ** -24  # unit round-off of FP32


def shifted(p, off):
    q = dict(p)
    for k in ("b0", "bf"):
        q[k] = np.array(p[k], dtype=float)
        q[k][:, 0] += off
    q["center"] = np.asarray(p["center"], dtype=float) + off
    return q


def same(a, b):
    for x, y in zip(a, b):
        if x is not None:
            np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("dims,mask", [(2, 7), (3, 7), (2, 1)])
@pytest.mark.parametrize("form", list(PER_SM))
@pytest.mark.parametrize("off,horizon", [(1e4, 6.0), (1e5, 1.0), (1e5, 6.0), (5e5, 2.0), (4.6e6, 5.0)])
def test_far_frames(P, oracle, off, horizon, form, dims, mask):  # noqa: F811
    """Frames up to a UTM northing.  Up to 100 km at 6 s against the oracle: FP32
    acceleration rows round by kappa u |offset| / T^2 (kappa: 81 with five free columns,
    630 with seven), which an iteration takes into the coefficients with a gain of
    at most sqrt(n_p dims) / 2: 17 and 130 u |offset|, 20 and 150 allowed in each of
    the K iterations on top of the usual tolerance."""
    p = shifted(scene(dims=dims, n_obs=24, n_dyn=3, n_p=60, horizon=horizon, mask=mask, amax=1.5), off)
    n = PER_SM[form] * sm_count() - 3
    xi = samples(oracle, p, n, seed=3)
    got = project(P, p, xi, K, None, "1")
    same(got, project(P, p, xi, K, None, "0"))
    xb, _, r, _ = got
    assert np.isfinite(xb).all() and np.isfinite(r).all()
    if off * (6.0 / horizon) ** 2 <= 1e5:
        idx = np.r_[0:n:max(1, n // 9), n - 1]
        xb_o, _ = oracle.project(p, xi[idx], K)
        assert np.abs(xb[idx] - xb_o).max() < TOL_FP32 * scale_of(p) + (20 if mask == 7 else 150) * K * U * off


@pytest.mark.parametrize("dims,mask", [(2, 7), (3, 7), (2, 1)])
@pytest.mark.parametrize("form", list(PER_SM))
@pytest.mark.parametrize("value", [1e9, -1e30])
def test_outlying_coefficients(P, oracle, value, form, dims, mask):  # noqa: F811
    """One coefficient of every fifth sample far off: the other samples are untouched."""
    p = scene(dims=dims, n_obs=24, n_dyn=3, n_p=60, mask=mask)
    n = PER_SM[form] * sm_count() - 3
    xi = samples(oracle, p, n, seed=3)
    odd = xi.copy()
    odd[::5, 5] = value
    a = project(P, p, odd, K, None, "1")
    same(a, project(P, p, odd, K, None, "0"))
    b = project(P, p, xi, K, None, "1")
    rest = np.arange(n) % 5 != 0
    for x, y in zip(a, b):
        if x is not None:
            np.testing.assert_array_equal(x[rest], y[rest])


@pytest.mark.parametrize("dims,mask", [(2, 7), (3, 7), (2, 1)])
@pytest.mark.parametrize("form", list(PER_SM))
def test_margin_below_resolution(P, oracle, form, dims, mask):  # noqa: F811
    p = scene(dims=dims, n_obs=24, n_dyn=3, n_p=60, mask=mask)
    n = PER_SM[form] * sm_count() - 3
    xi = samples(oracle, p, n, seed=3)
    os.environ["PRIEST_LIST_MARGIN"] = "1e-8"
    try:
        a = project(P, p, xi, K, None, "1")
    finally:
        os.environ.pop("PRIEST_LIST_MARGIN")
    same(a, project(P, p, xi, K, None, "0"))
