"""A walk gives the same numbers however many lanes run it: a lane alone (the
mixed walk in a launch that fills the GPU), four lanes (the double-precision
walk there), or all the lanes of a warp (a launch of few walks).  The same
paths from both, over the densities, domains and options of either walk, path
counts that leave ragged groups, and step caps inside a block."""
import numpy as np
import pytest
import torch

import oracle
from paper_1709_07469_gb300 import build as B
from paper_1709_07469_gb300 import mcgrav as M
from paper_1709_07469_gb300 import workloads as W
from paper_1709_07469_gb300.device import DeviceSolve
from tests.helpers import smooth_tables

pytestmark = pytest.mark.gpu
FULL = {M.MCG_MIXED: 200_000, M.MCG_FP64: 20_000}  # walks that fill the GPU
BOTH = pytest.mark.parametrize("precision", [M.MCG_MIXED, M.MCG_FP64])


@pytest.fixture(scope="module", autouse=True)
def lib():
    B.build()
    M.load()


def per_path(w, st, N, cap, **kw):
    ds = DeviceSolve(w, stations=st, batch=N, **kw)
    if cap:
        ds.opts.max_steps = cap
    ds.reset()
    ds.walk(0)
    return (*ds.per_path(), int(ds.status[0].item()))


def same_paths(w, few, precision, cap=None, rounding=0.0, **kw):
    st = w.stations[:2]
    a = per_path(w, st, few, cap, precision=precision, **kw)
    b = per_path(w, st, FULL[precision] // 2, cap, precision=precision, **kw)
    assert a[3] == b[3]
    assert np.array_equal(a[2], b[2][:, :few])
    for x, y in zip(a[:2], b[:2]):
        y = y[:, :few]
        assert np.array_equal(np.isnan(x), np.isnan(y))
        if rounding:
            ok = ~np.isnan(x)
            scale = np.abs(b[0][:, :few][ok]).max()
            np.testing.assert_allclose(x[ok], y[ok], rtol=0, atol=rounding * scale)
        else:
            assert np.array_equal(x, y, equal_nan=True)


SPHERE = W.sphere_line()
CASES = {
    "sphere": SPHERE,
    "prism": W.prism_ore_body(step=10.0),
    "none": W.unit_box(SPHERE.stations, g_kind="poly", poly=(0, 0, 0, 0, 1.0, 1.0, -2.0, 0, 0, 0, 0), dt=1e-3),
    "ball": W.paper_cube_ball(step=200.0),
    "bridge": SPHERE.with_(bridge=1, dt=4e-3),
    "plain": W.prism_ore_body(step=10.0).with_(crn=0),
}


@BOTH
@pytest.mark.parametrize("few", [1, 5, 33, 1001])
@pytest.mark.parametrize("name", CASES)
def test_shared_walks_equal_lone_ones(name, few, precision):
    same_paths(CASES[name], few, precision)


@BOTH
@pytest.mark.parametrize("cap", [1, 6, 127, 130])
def test_step_cap_inside_a_shared_round(cap, precision):
    same_paths(SPHERE.with_(dt=4e-3), 9, precision, cap=cap)


@pytest.mark.parametrize("precision,pack", [(M.MCG_MIXED, True), (M.MCG_MIXED, False), (M.MCG_FP64, False)])
@pytest.mark.parametrize("few", [1, 7, 300])
def test_shared_walks_voxel(few, precision, pack):
    """Single-precision partial sums: the flush points of a lane's walk follow
    its warp's refills, so u may differ by the rounding of one flush, at most
    64 * 2^-24 ~ 4e-6 of the source integral, which is below max |u| here (and
    u by 1 / h of that in the centred difference, h = 1).  The double-precision
    walk's sums are added per lane, then over the lanes: up to 4000 terms in
    another order, 4000 * 2^-53 < 1e-12."""
    w = W.voxel_survey(shape=(32, 32, 16), table_n=(33, 33), step=20.0)
    grid = torch.from_numpy(oracle.grf_density(1, 32, 32, 16, sigma_vox=2.0, amp=300.0)).cuda()
    faces = torch.from_numpy(smooth_tables(w, scale=-1e-4)).cuda()
    rounding = 4e-6 if precision == M.MCG_MIXED else 1e-12
    same_paths(w, few, precision, rounding=rounding, grid=grid, faces=faces, pack=pack)
