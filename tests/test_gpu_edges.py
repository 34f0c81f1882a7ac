"""Calls at the ends of what the entry points accept, and after an error.

* step cap: the largest integer is no cap at all;
* double-precision normals: every digit of the small ones too;
* a density that is not finite: only the walks that meet it;
* boundary tables: grids of many cells in a row; near zones of a few cells;
* the field of small grids to the last digits that doubles hold; of long ones;
* an error of one launch is not reported by the next;
* mcgrav_solve: its workspace goes back, and a failed call waits as well;
* mcgrav_solve after a device reset;
"""
import ctypes
import os
import subprocess
import sys

import numpy as np
import pytest
import torch

import oracle
from paper_1709_07469_gb300 import build as B
from paper_1709_07469_gb300 import mcgrav as M
from paper_1709_07469_gb300 import workloads as W
from paper_1709_07469_gb300.device import DeviceSolve
from tests.helpers import oracle_spec

pytestmark = pytest.mark.gpu
THREADS = os.cpu_count() or 1


@pytest.fixture(scope="module", autouse=True)
def lib():
    B.build()
    M.load()


@pytest.mark.parametrize("precision", [M.MCG_FP64, M.MCG_MIXED])
@pytest.mark.parametrize("cap", [2**63 - 1, 2**63 - 4])
def test_largest_step_cap_caps_nothing(precision, cap):
    w = W.sphere_line(paths=64)
    out = []
    for c in (1 << 31, cap):
        ds = DeviceSolve(w, stations=w.stations[:2], precision=precision)
        ds.opts.max_steps = c
        ds.reset()
        ds.walk(0)
        assert int(ds.status[0].item()) == 0
        out.append(ds.per_path())
    for a, b in zip(*out):
        assert np.array_equal(a, b)


def test_fp64_normals_keep_their_leading_digits():
    """Relative to themselves, also the small ones (a radius next to 0, an angle
    next to an axis).  In units of 2^-52: here 1 for the radius (logarithm 1,
    halved by the root, its rounding 1/2), 2 for cosine or sine, 1/2 for the
    product; the host's 1/2 or less each of logarithm (halved), root, product, and
    1 of cosine or sine: 6 in all with the rest for second order."""
    nb = 1 << 17
    out = torch.empty(12 * nb, dtype=torch.float64, device="cuda")
    M.mcg_normals(11, 3, 5, 0, nb, M.MCG_FP64, out)
    got, want = out.cpu().numpy(), oracle.normals(11, 3, 5, 0, nb)
    assert np.abs(want).min() < 1e-5
    assert np.all(np.abs(got - want) <= 6 * 2.0**-52 * np.abs(want))


def box_of_cells(shape, side, air=0.0):
    """A voxel workload whose domain is its grid of cubes, `air` more above it."""
    n = np.array(shape, dtype=np.float64) * side
    w = W.voxel_survey(shape=shape).with_(g_kind="zero", G=1.0)
    return w.with_(lo=tuple(-0.5 * n), hi=tuple(0.5 * n + np.array([0.0, 0.0, air])), grid_origin=tuple(-0.5 * n),
                   grid_spacing=(side, side, side))


@pytest.mark.parametrize("shape", [(1, 3000, 1), (2, 20000, 1), (1, 200000, 1), (1, 1, 20000)])
def test_tables_of_long_thin_grids(shape):
    """A near zone over a grid of up to 2e5 cells in a row.  Reference: direct
    prism sums of the 64 cells next to the node's end (beyond, they cancel), point
    masses in doubles for the others (a cube's next term: 0.2 (1 / 128)^4 of its
    own).  Result rounded to single precision, allowance 3e-7 as in
    test_gpu_setup.py."""
    w = box_of_cells(shape, 10.0)
    axis = int(np.argmax(shape))
    rng = np.random.default_rng(axis)
    grid = rng.uniform(100.0, 500.0, shape[::-1]).astype(np.float32)
    faces = torch.empty((6, 2, 2), dtype=torch.float32, device="cuda")
    M.mcg_boundary_tables(M.problem(w, grid=torch.from_numpy(grid).cuda()), 2, 2, 1e6, faces)
    got = faces.cpu().numpy().astype(np.float64)
    fi, iv, iu = np.meshgrid(np.arange(6), np.arange(2), np.arange(2), indexing="ij")
    lo, hi = np.array(w.lo), np.array(w.hi)
    sp = np.array(w.grid_spacing)
    along = np.arange(shape[axis])
    to = [1] * 3
    to[2 - axis] = -1
    ends = []
    for first in (along < 64, along >= shape[axis] - 64):
        near = np.where(first.reshape(to), grid, 0).astype(np.float32)
        ends.append((oracle.table_nodes(oracle_spec(w, grid=near), fi.ravel(), iu.ravel(), iv.ravel(), 2, 2,
                                        threads=THREADS), np.where(first.reshape(to), 0.0, grid.astype(np.float64))))
    c = [(lo[k] + (np.arange(shape[k]) + 0.5) * sp[k]).reshape([-1 if 2 - k == d else 1 for d in range(3)])
         for k in range(3)]
    for e, (f, b, a) in enumerate(zip(fi.ravel(), iv.ravel(), iu.ravel())):
        k = f // 2
        p, q = [(1, 2), (0, 2), (0, 1)][k]
        x = np.zeros(3)
        x[k], x[p], x[q] = (hi if f % 2 else lo)[k], (hi if a else lo)[p], (hi if b else lo)[q]
        exact, far = ends[0 if x[axis] < 0.0 else 1]
        r = np.sqrt((c[0] - x[0]) ** 2 + (c[1] - x[1]) ** 2 + (c[2] - x[2]) ** 2)
        want = exact[e] - w.G * np.prod(sp) * np.sum(far / r)
        np.testing.assert_allclose(got[f, b, a], want, rtol=3e-7)


@pytest.mark.parametrize("near", [1.5, 2.0, 3.0])
def test_tables_of_a_cell_at_the_rim_of_a_small_near_zone(near):
    """A dense cell two to four of its sides below a node: its own prism potential,
    rounded to single precision (half a unit in the last place; the sums before
    are doubles: 1e-3 of one more)."""
    w = box_of_cells((1, 1, 1), 1.0)
    grid = torch.full((1, 1, 1), 500.0, dtype=torch.float32, device="cuda")
    faces = torch.empty((6, 3, 3), dtype=torch.float32, device="cuda")
    gaps = np.linspace(1.5, min(near * np.sqrt(3.0), 4.2) - 0.51, 200)
    for gap in gaps:
        v = w.with_(hi=(0.5, 0.5, 0.5 + gap))
        M.mcg_boundary_tables(M.problem(v, grid=grid), 3, 3, near, faces)
        got = faces[5, 1, 1].item()
        want = oracle.prism_phi(1.0, 500.0, (-0.5, -0.5, -0.5), (0.5, 0.5, 0.5), (0.0, 0.0, 0.5 + gap))
        assert abs(got - want) <= 0.501 * np.spacing(np.float32(abs(want))), gap


@pytest.mark.parametrize("precision", [M.MCG_FP64, M.MCG_MIXED])
@pytest.mark.parametrize("rho0", [float("inf"), float("nan")])
@pytest.mark.parametrize("kind", ["prism", "sphere"])
def test_nonfinite_density_reaches_only_the_walks_that_meet_it(precision, rho0, kind):
    """With zero boundary data a walk that never met the body has u = 0 for any
    density of the body; only the others are lost to a density that is not finite."""
    w = W.prism_ore_body(paths=512, step=20.0) if kind == "prism" else W.sphere_line(paths=512)
    st = w.stations[:1] if kind == "prism" else np.array([[0.0, 0.0, 0.9]])
    w = w.with_(g_kind="zero", stations=st)
    met = None
    for r in (w.rho0, rho0):
        ds = DeviceSolve(w.with_(rho0=r), precision=precision)
        ds.reset()
        ds.walk(0)
        u = ds.per_path()[0]
        status = int(ds.status[0].item())
        if met is None:
            met = u != 0.0
            assert 0 < met.sum() < met.size and status == 0
        else:
            assert np.all(u[~met] == 0.0)
            assert not np.any(np.isfinite(u[met]))
            assert status == 1 << M.MCG_ERR_NONFINITE


def invalid_stream():
    """A stream whose capture has been broken: whatever is launched into it is
    refused.  Returns (stream, end): nothing is left of it after end()."""
    cu = ctypes.CDLL("libcuda.so.1")
    st = ctypes.c_void_p()
    assert cu.cuStreamCreate(ctypes.byref(st), 1) == 0
    assert cu.cuStreamBeginCapture_v2(st, 2) == 0          # (relaxed: other streams are not concerned)
    assert cu.cuStreamSynchronize(st) != 0                 # not allowed in a capture: ends it with an error

    def end():
        graph = ctypes.c_void_p()
        assert cu.cuStreamEndCapture(st, ctypes.byref(graph)) != 0
        assert cu.cuStreamDestroy_v2(st) == 0

    return st.value, end


@pytest.mark.parametrize("call", ["field", "tables"])
def test_a_refused_launch_leaves_no_error_behind(call):
    w, grid = box_of_cells((4, 4, 4), 1.0), torch.ones((4, 4, 4), dtype=torch.float32, device="cuda")
    prob = M.problem(w, grid=grid)
    x = torch.full((1, 3), 5.0, dtype=torch.float64, device="cuda")
    phi = torch.empty(1, dtype=torch.float64, device="cuda")
    faces = torch.empty((6, 2, 2), dtype=torch.float32, device="cuda")

    def field(stream):
        M.mcg_field(prob, x, 1, phi, None, stream)

    def tables(stream):
        M.mcg_boundary_tables(prob, 2, 2, 4.0, faces, stream)

    torch.cuda.synchronize()
    st, end = invalid_stream()
    try:
        with pytest.raises(M.McgError):
            (field if call == "field" else tables)(st)
    finally:
        end()
    for good in (tables, field):
        good(None)
    torch.cuda.synchronize()
    assert np.isfinite(phi.item()) and np.all(np.isfinite(faces.cpu().numpy()))


def used_bytes():
    free, total = torch.cuda.mem_get_info()
    return total - free


def test_solve_hands_its_workspace_back():
    """At most 256 MiB of a solve's workspace stay with the library after the
    call, without a further synchronisation."""
    w = W.sphere_line(dt=0.04)
    opts = M.options(w, batch_paths=1 << 18)
    M.mcgrav_solve(M.problem(w), w.stations, 64, w.dt, 0, M.options(w))
    torch.cuda.synchronize()
    before = used_bytes()
    assert M.mcg_workspace_bytes(8, 1 << 18) > (512 << 20)
    M.mcgrav_solve(M.problem(w), w.stations, 1 << 19, w.dt, 0, opts)
    assert used_bytes() - before <= 256 << 20


def test_a_failed_solve_waits_for_its_copies():
    """A grid of one layer too large to pack is refused after its copy to the
    device has been queued: the call returns once the copy is done, as the
    caller's (pinned) array may go away then."""
    nx, ny = 1 << 15, (1 << 31) // 3 // (1 << 15) + 1
    w = box_of_cells((8, 8, 8), 10.0).with_(g_kind="zero", stations=np.zeros((1, 3)), paths=1)
    grid = torch.empty((1, ny, nx), dtype=torch.float32, pin_memory=True)
    prob = M.problem(w, grid=grid.numpy())
    st = torch.cuda.Stream()
    r = M.mcgrav_solve(prob, w.stations, 1, w.dt, 0, M.options(w, stream=st), allow=(M.MCG_ERR_ARG,))
    assert st.query()
    assert r.status == M.MCG_ERR_ARG and "too large to pack" in M.last_error()


RESET = """
import ctypes, os
import numpy as np
from paper_1709_07469_gb300 import mcgrav as M, workloads as W

M.load()
w = W.sphere_line(dt=0.01)


def solve():
    return M.mcgrav_solve(M.problem(w), w.stations, 64, w.dt, 0, M.options(w)).u


first = solve()
for _ in range(3):
    assert ctypes.CDLL(os.environ["CUDART"]).cudaDeviceReset() == 0
    for _ in range(2):
        assert np.array_equal(solve(), first)
"""


def cudart():
    with open("/proc/self/maps") as f:
        found = {line.split()[-1] for line in f if "libcudart.so" in line}
    return found.pop()


def test_solve_after_a_device_reset():
    """The program's own runtime resets the device (its process alone is
    concerned): the library takes up a new context."""
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", RESET], cwd=root, env=dict(os.environ, CUDART=cudart(), PYTHONPATH=root),
                       capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stderr


def field_in_long_doubles(w, grid, points):
    """dPhi/dz by node sums in numpy's long doubles (64-bit mantissa or more), and
    the sum of the cells' own magnitudes."""
    L = np.longdouble
    nz, ny, nx = grid.shape
    weight = np.zeros((nz + 1, ny + 1, nx + 1), L)
    for m in range(8):
        i, j, k = m & 1, m >> 1 & 1, m >> 2
        weight[k:k + nz, j:j + ny, i:i + nx] += grid.astype(L) * (1 if (i + j + k) & 1 else -1)
    x, y, z = (L(w.grid_origin[a]) + np.arange(n + 1, dtype=L) * L(w.grid_spacing[a]) for a, n in
               enumerate((nx, ny, nz)))
    gz, size = [], []
    for p in points:
        a, b, c = (x - L(p[0]))[None, None, :], (y - L(p[1]))[None, :, None], (z - L(p[2]))[:, None, None]
        r = np.sqrt(a * a + b * b + c * c)

        def ln(t, s2):      # ln(t + r), without cancellation
            t = t + 0 * r
            return np.where(t < 0, np.log(s2 + 0 * r) - np.log(r + np.abs(t)), np.log(r + np.abs(t)))

        D = a * ln(b, a * a + c * c) + b * ln(a, b * b + c * c) - c * np.arctan(a * b / (c * r))
        gz.append(float(w.G * np.sum(weight * D)))
        mid = [(v[1:] + v[:-1]) / 2 for v in (a.ravel(), b.ravel(), c.ravel())]
        r2 = mid[0][None, None, :] ** 2 + mid[1][None, :, None] ** 2 + mid[2][:, None, None] ** 2
        size.append(float(w.G * np.prod(w.grid_spacing) * np.sum(np.abs(grid) / r2)))
    return np.array(gz), np.array(size)


@pytest.mark.parametrize("shape", [(20, 17, 9), (16, 16, 8), (31, 19, 8)])
def test_field_of_small_grids_over_their_surface(shape):
    """Where single-precision terms of few cells weigh most.  Bound: 3e-14 for the
    pairs (2^-45 of every cell), 1.2e-13 for the cancellation of the near nodes in
    doubles (their terms are some 500 times the cells'), 5e-14 for what remains of
    the series (1e-12 of the cells beyond the rim, a twentieth of the sum)."""
    w = W.voxel_survey(shape=shape).with_(g_kind="zero")
    rng = np.random.default_rng(5)
    grid = (300.0 * np.expm1(rng.normal(size=shape[::-1]))).astype(np.float32)
    pts = rng.uniform(w.lo, w.hi, (40, 3))
    pts[:, 2] = 0.01 * np.abs(pts[:, 2])
    out = torch.empty((2, 40), dtype=torch.float64, device="cuda")
    M.mcg_field(M.problem(w, grid=torch.from_numpy(grid).cuda()), torch.from_numpy(pts).cuda(), 40, out[0], out[1])
    want, size = field_in_long_doubles(w, grid, pts)
    assert np.all(np.abs(out[1].cpu().numpy() - want) <= 2e-13 * size)


@pytest.mark.parametrize("shape", [(1, 20000, 1), (1, 65534, 1), (40000, 1, 2)])
def test_field_of_long_grids(shape):
    """Rows of up to 65534 cubes, points over and beside them.  Reference: prism
    sums for the cells within 64 sides, point masses for the others (the next term
    of a cube: 0.2 (1 / 128)^4 of its own, 1e-9)."""
    w = box_of_cells(shape, 10.0)
    axis = int(np.argmax(shape))
    grid = np.random.default_rng(axis).uniform(100.0, 500.0, shape[::-1]).astype(np.float32)
    pts = np.zeros((12, 3))
    pts[:, axis] = 10.0 * np.array([0.0, 3.3, 7000.4, -0.5 * shape[axis] + 2.0] * 3)
    pts[:, 2] += np.repeat([12.0, 71.0, 300.0], 4)
    out = torch.empty((2, 12), dtype=torch.float64, device="cuda")
    M.mcg_field(M.problem(w, grid=torch.from_numpy(grid).cuda()), torch.from_numpy(pts).cuda(), 12, out[0], out[1])
    got = out.cpu().numpy()
    c = [(w.lo[k] + 10.0 * (np.arange(shape[k]) + 0.5)).reshape([-1 if 2 - k == d else 1 for d in range(3)])
         for k in range(3)]
    to = [1] * 3
    to[2 - axis] = -1
    for i, x in enumerate(pts):
        near = np.abs(c[axis].ravel() - x[axis]) < 640.0
        part = np.where(near.reshape(to), grid, 0).astype(np.float32)
        phi, gz = oracle.voxel_field(oracle_spec(w, grid=part), x[None, :], threads=THREADS, want_gz=True)
        far = np.where(near.reshape(to), 0.0, grid.astype(np.float64))
        r = np.sqrt((c[0] - x[0]) ** 2 + (c[1] - x[1]) ** 2 + (c[2] - x[2]) ** 2)
        np.testing.assert_allclose(got[0, i], phi[0] - w.G * 1000.0 * np.sum(far / r), rtol=1e-8)
        np.testing.assert_allclose(got[1, i], gz[0] - w.G * 1000.0 * np.sum(far * (c[2] - x[2]) / r**3), rtol=1e-8)
