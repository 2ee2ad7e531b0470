"""The FP32 point-owner projection at the limits of its inputs and lists, in every form
(teams of four and of two warps per sample, one warp, two samples per warp): bitwise the
results of screening every pair in every iteration."""
import os
from math import comb

import numpy as np
import pytest

from gpu_common import samples, scene
from paper_2309_08235_gb300 import workloads as W
from test_gpu_pts_edges import P, PER_SM, project, sm_count  # noqa: F401
from test_gpu_pts_frames import same

pytestmark = pytest.mark.gpu

FORMS = pytest.mark.parametrize("form", list(PER_SM))
SHAPES = pytest.mark.parametrize("dims,mask", [(2, 7), (3, 7), (2, 1)])


@SHAPES
@FORMS
@pytest.mark.parametrize("bounds", [False, True])
def test_coefficient_turns_nan(P, oracle, bounds, form, dims, mask):  # noqa: F811
    """A multiplier beyond FP32's range makes one axis infinite, then NaN, after the lists
    were built: what that does to the other axes is the same with lists and without,
    and other samples are untouched."""
    p = scene(dims=dims, n_obs=12, n_dyn=2, n_p=60, mask=mask, bounds=bounds, vmax=30.0, amax=60.0)
    n = PER_SM[form] * sm_count() - 3
    xi = samples(oracle, p, n, seed=3)
    lam0 = np.zeros_like(xi)
    good = project(P, p, xi, 8, lam0, "1")
    odd = lam0.copy()
    odd[::5, 5] = 1e300
    got = project(P, p, xi, 8, odd, "1")
    same(got, project(P, p, xi, 8, odd, "0"))
    assert np.isnan(got[0][::5]).any(axis=1).all()
    rest = np.arange(n) % 5 != 0
    for x, y in zip(got, good):
        np.testing.assert_array_equal(x[rest], y[rest])


@pytest.mark.parametrize("dims", [2, 3])
@FORMS
def test_next_to_the_centre(P, oracle, form, dims):  # noqa: F811
    """A robot at rest within 1e-18 of an obstacle's centre: squared offsets are denormal
    in FP32, the push is the semi-axis all the same.  One iteration; a denormal square of
    1e-40 holds five digits, those below 1e-43 belong to the time stamps next to the
    ends, whose rows weigh less than 1e-3: 5e-3 of the largest push allowed."""
    p = scene(dims=dims, n_obs=1, n_dyn=0, n_p=60, radius=(1.0, 1.0), vmax=1e6, amax=1e6)
    p = dict(p, center=np.zeros((1, dims)), b0=np.zeros((dims, 3)), bf=np.zeros((dims, 3)))
    n = PER_SM[form] * sm_count() - 3
    rng = np.random.default_rng(5)
    xi = np.zeros((n, dims, 11))
    xi[:, :, 3:8] = 1e-19 * (rng.choice([-1.0, 1.0], (n, dims, 1)) + 0.1 * rng.normal(size=(n, dims, 5)))
    xi = xi.reshape(n, -1)
    got = project(P, p, xi, 1, None, "1")
    same(got, project(P, p, xi, 1, None, "0"))
    idx = np.r_[0:n:max(1, n // 20), n - 1]
    xb_o, _ = oracle.project(p, xi[idx], 1)
    assert np.abs(xb_o).max() > 0.01
    assert np.abs(got[0][idx] - xb_o).max() < 5e-3 * np.abs(xb_o).max()


def near_pairs(p, xb, grow):
    """Per sample, the (time stamp, obstacle) pairs within `grow` semi-axes."""
    dims, n_p = p["dims"], p["n_p"]
    tau = np.arange(n_p) / (n_p - 1)
    B = np.stack([comb(10, j) * tau ** j * (1 - tau) ** (10 - j) for j in range(11)], 1)
    x = np.einsum("tj,naj->nta", B, np.asarray(xb).reshape(len(xb), dims, 11))
    o = np.asarray(p["center"]) + (tau * p["horizon"])[:, None, None] * np.asarray(p["vel"])
    s = np.asarray(p["semi"])[:, [0, 0, 1][:dims]]
    d = (x[:, :, None, :] - o) / s
    return np.count_nonzero((d * d).sum(3) < grow * grow, axis=(1, 2))


def crowd(dims, mask, kind):
    if kind == "pile":  # every time stamp inside several obstacles, to the end
        return scene(dims=dims, n_obs=40, n_dyn=5, n_p=70, mask=mask, radius=(3.0, 5.0))
    # forty obstacles on one spot of the straight line, which the samples leave
    p = scene(dims=dims, n_obs=40, n_dyn=0, n_p=70, mask=mask)
    mid = 0.5 * (np.asarray(p["b0"])[:, 0] + np.asarray(p["bf"])[:, 0])
    return dict(p, center=np.tile(mid, (40, 1)), semi=np.full((40, 2), 1.4), vel=np.zeros((40, dims)))


K_LONG = 48  # three times the iterations after which a list that overflowed is tried again


@pytest.mark.parametrize("kind", ["pile", "cleared"])
@SHAPES
@FORMS
def test_lists_overflow_and_return(P, oracle, kind, form, dims, mask):  # noqa: F811
    """More pairs than a list holds (256), for good or until the samples have moved
    away, over several of the tries at a new list: bitwise as without lists."""
    p = crowd(dims, mask, kind)
    n = PER_SM[form] * sm_count() - 3
    xi = samples(oracle, p, n, seed=3, std=0.3)
    idx = np.r_[0:n:max(1, n // 9), n - 1]
    assert (near_pairs(p, oracle.project_eq(p, xi[idx]), 1.0) > 256).all()
    if kind == "cleared":
        assert (near_pairs(p, oracle.project(p, xi[idx], 16)[0], 2.5) <= 256).all()
    same(project(P, p, xi, K_LONG, np.zeros_like(xi), "1"), project(P, p, xi, K_LONG, np.zeros_like(xi), "0"))


def test_default_margin_changes_no_bit(P, oracle):  # noqa: F811
    """The margin set by the obstacles' density against a fixed one."""
    p = W.scene_clutter_2d(seed=3, n_static=90, n_dyn=10, n_p=100)
    xi = oracle.default_mean(p) + 2.0 * W.normals(77, (300, 22))
    lam0 = np.random.default_rng(8).normal(0.0, 0.1, xi.shape)
    got = project(P, p, xi, 40, lam0, "1")
    os.environ["PRIEST_LIST_MARGIN"] = "0.75"
    try:
        same(got, project(P, p, xi, 40, lam0, "1"))
    finally:
        os.environ.pop("PRIEST_LIST_MARGIN")


@SHAPES
@FORMS
def test_margin_beyond_range(P, oracle, form, dims, mask):  # noqa: F811
    """Semi-axes whose margin overflows FP32, every pair near: the lists overflow at
    every margin, and halving it ends."""
    p = scene(dims=dims, n_obs=40, n_dyn=4, n_p=60, mask=mask)
    p = dict(p, semi=np.full((40, 2), 2e38))
    n = PER_SM[form] * sm_count() - 3
    xi = samples(oracle, p, n, seed=3)
    got = project(P, p, xi, 8, None, "1")
    assert got[0].shape == xi.shape
    same(got, project(P, p, xi, 8, None, "0"))
