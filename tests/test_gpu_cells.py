"""The cell series behind mcg_field and mcg_boundary_tables against the
oracle's direct prism sums: cells that are not cubes, grids thinner than a
block's tile or wider than it by a ragged rest, points near, inside and far
from the grid, and the launch shapes for few and many points or nodes.

Tolerances: the field is a double-precision sum; the oracle's direct sum of
prisms cancels to about 1e-11 of itself at these sizes (as in
test_gpu_field.py: 1e-10).  Tables whose near zone covers the grid are the
exact sum rounded to single precision (6e-8, allowance 3e-7 as in
test_gpu_setup.py)."""
import os

import numpy as np
import pytest
import torch

import oracle
from paper_1709_07469_gb300 import build as B
from paper_1709_07469_gb300 import mcgrav as M
from paper_1709_07469_gb300 import workloads as W
from tests.helpers import oracle_spec

pytestmark = pytest.mark.gpu
THREADS = os.cpu_count() or 4


@pytest.fixture(scope="module", autouse=True)
def lib():
    B.build()
    M.load()


def model(shape, table=9):
    w = W.voxel_survey(shape=shape, table_n=(table, table)).with_(g_kind="zero")
    grid = np.random.default_rng(sum(shape)).uniform(-100.0, 500.0, shape[::-1]).astype(np.float32)
    return w, grid


SHAPES = [(1, 1, 1), (3, 40, 2), (17, 5, 9), (33, 4, 3), (16, 16, 8)]


@pytest.mark.parametrize("shape", SHAPES)
def test_field_of_any_cell_shape(shape):
    w, grid = model(shape)
    rng = np.random.default_rng(1)
    pts = np.concatenate([rng.uniform(w.lo, w.hi, (20, 3)), [[0.0, 0.0, 0.0], [0.0, 0.0, 5000.0], [3e5, -1e5, 2e5]]])
    n = len(pts)
    out = torch.empty((2, n), dtype=torch.float64, device="cuda")
    M.mcg_field(M.problem(w, grid=torch.from_numpy(grid).cuda()), torch.from_numpy(pts).cuda(), n, out[0], out[1])
    phi, gz = out.cpu().numpy()
    ref_phi, ref_gz = oracle.voxel_field(oracle_spec(w, grid=grid), pts[:-1], threads=THREADS, want_gz=True)
    np.testing.assert_allclose(phi[:-1], ref_phi, rtol=1e-10)
    np.testing.assert_allclose(gz[:-1], ref_gz, rtol=1e-9, atol=1e-9 * np.abs(ref_gz).max())
    # far away the direct sum has cancelled: there the cells are point masses
    # up to (cell / distance)^2 ~ 1e-4 of their quadrupole
    c = np.stack(np.meshgrid(*[np.array(w.grid_origin)[k] + (np.arange(shape[k]) + 0.5) * w.grid_spacing[k]
                               for k in range(3)], indexing="ij"), -1).transpose(2, 1, 0, 3)
    r = np.linalg.norm(c - pts[-1], axis=-1)
    want = -w.G * np.prod(w.grid_spacing) * np.sum(grid.astype(np.float64) / r)
    np.testing.assert_allclose(phi[-1], want, rtol=1e-4)


def test_field_of_many_points_equals_that_of_few():
    w, grid = model((17, 5, 9))
    prob = M.problem(w, grid=torch.from_numpy(grid).cuda())
    pts = torch.from_numpy(np.random.default_rng(2).uniform(w.lo, w.hi, (2100, 3))).cuda()
    many = torch.empty((2, 2100), dtype=torch.float64, device="cuda")
    few = torch.empty((2, 3), dtype=torch.float64, device="cuda")
    M.mcg_field(prob, pts, 2100, many[0], many[1])
    M.mcg_field(prob, pts, 3, few[0], few[1])
    # other partial sums of the same terms: rounding only
    np.testing.assert_allclose(many[:, :3].cpu(), few.cpu(), rtol=1e-11)


@pytest.mark.parametrize("shape,table,near", [((3, 40, 2), 5, 1e6), ((17, 5, 9), 5, 1e6), ((16, 16, 8), 81, 1e6),
                                              ((16, 16, 8), 81, 1.0), ((7, 9, 4), 33, 2.0)])
def test_tables_of_any_cell_shape(shape, table, near):
    """near = 1e6 covers the grid; smaller near zones leave point masses, whose
    error is compared with that of the same split evaluated in numpy."""
    w, grid = model(shape, table)
    faces = torch.empty((6, table, table), dtype=torch.float32, device="cuda")
    M.mcg_boundary_tables(M.problem(w, grid=torch.from_numpy(grid).cuda()), table, table, near, faces)
    f = faces.cpu().numpy()
    rng = np.random.default_rng(3)
    fi, iu, iv = rng.integers(0, 6, 60), rng.integers(0, table, 60), rng.integers(0, table, 60)
    spec = oracle_spec(w, grid=grid)
    want = oracle.table_nodes(spec, fi, iu, iv, table, table, threads=THREADS)
    got = f[fi, iv, iu].astype(np.float64)
    if near < 1e6:
        # every voxel's point mass, and which of them the near zone replaces
        sp, org = np.array(w.grid_spacing), np.array(w.grid_origin)
        c = np.stack(np.meshgrid(*[org[k] + (np.arange(shape[k]) + 0.5) * sp[k] for k in range(3)], indexing="ij"),
                     -1).transpose(2, 1, 0, 3)
        for i in range(60):
            k = fi[i] // 2
            a, b = [(1, 2), (0, 2), (0, 1)][k]
            x = np.zeros(3)
            x[k] = (w.hi if fi[i] % 2 else w.lo)[k]
            x[a] = w.lo[a] + (w.hi[a] - w.lo[a]) * iu[i] / (table - 1)
            x[b] = w.lo[b] + (w.hi[b] - w.lo[b]) * iv[i] / (table - 1)
            r = np.linalg.norm(c - x, axis=-1)
            far = r >= near * np.linalg.norm(sp)
            g = np.where(far, grid, 0).astype(np.float32)
            exact_far = oracle.table_nodes(oracle_spec(w, grid=g), fi[i:i + 1], iu[i:i + 1], iv[i:i + 1], table, table)
            want[i] += -w.G * np.prod(sp) * np.sum(g.astype(np.float64) / r) - exact_far[0]
        # single-precision point masses: some 1e-7 each, of either sign
        np.testing.assert_allclose(got, want, rtol=2e-6, atol=1e-6 * np.abs(want).max())
    else:
        np.testing.assert_allclose(got, want, rtol=3e-7, atol=1e-7 * np.abs(want).max())
