"""Pressure loads at the edges of the load kernel's lists: a hub node in
fewer, exactly and more than 32 triangles (one list), triangle counts around
the 128 scanned together, node counts that leave warps of the last block
idle, and nodes near and beyond the box faces (periodic interpolation).
Tolerance: FP64 sums of at most 216 points and 129 triangles, 1e-12 of the
largest value.
"""
import math

import numpy as np
import pytest
import torch

from oracle import mask as OM
from oracle import pressure as OP
from paper_2002_08642_gb300 import build as pbuild
from paper_2002_08642_gb300 import inputs
from paper_2002_08642_gb300.solver import Solver

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    pbuild.build()


@pytest.mark.parametrize("rim,nz", [(3, 32), (32, 32), (33, 16), (70, 32), (127, 32), (129, 16)])
def test_loads_of_a_fan(rim, nz):
    n, L = 32, 4.0
    th = 2.0 * math.pi * np.arange(rim) / rim
    xw = np.concatenate([[[0.05, -0.1, 0.02]], np.stack([np.cos(th), np.sin(th), 0.3 * np.cos(2 * th)], axis=1)])
    tri = np.asarray([(0, 1 + i, 1 + (i + 1) % rim) for i in range(rim)], dtype=np.int32)
    fr = inputs.frame(inputs.rot_z(0.7) @ inputs.rot_y(25.0), (0.9, 3.4, 1.9))   # some nodes outside the box
    p = np.random.default_rng(rim).standard_normal((n, n, nz))
    g = Solver(n, L, 1e-3, 1e-3, 5e-4, precision="fp64", nz=nz)
    d = lambda a, t: torch.from_numpy(np.ascontiguousarray(a)).to("cuda", t)
    pn, fn = g.pressure_loads(d(p, torch.float64), d(xw, torch.float64), d(tri, torch.int32), fr)
    xg = OM.global_nodes(xw, fr)
    pn_o = OP.interpolate(p, L, xg)
    fn_o = OP.node_loads(pn_o, xg, tri)
    assert np.abs(pn.cpu().numpy() - pn_o).max() < 1e-12 * np.abs(pn_o).max()
    assert np.abs(fn.cpu().numpy() - fn_o).max() < 1e-12 * np.abs(fn_o).max()
