"""Calls at the ends of what the entry points accept, and after an error.

* step cap: the largest integer is no cap at all;
"""
import numpy as np
import pytest
import torch

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
