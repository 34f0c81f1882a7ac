"""Calls at the ends of what the entry points accept, and after an error.

* step cap: the largest integer is no cap at all;
* double-precision normals: every digit of the small ones too;
"""
import numpy as np
import pytest
import torch

import oracle
from paper_1709_07469_gb300 import build as B
from paper_1709_07469_gb300 import mcgrav as M
from paper_1709_07469_gb300 import workloads as W
from paper_1709_07469_gb300.device import DeviceSolve

pytestmark = pytest.mark.gpu


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
