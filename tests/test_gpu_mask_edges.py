"""The rasteriser at the edges of its work split: a box of fewer points than a
warp, two large triangles (many warps each), more triangles than warps are
asked for, boxes cut by the grid's faces, slivers, an n x n x n/2 grid, and a
second call on the same context that clears the first. chi against the oracle
(1e-12 in FP64, 2e-6 in FP32, as for the wing); the node velocities are a
rigid rotation, so that u_s is the same whichever of two equally close
triangles wins: 1e-12 of its largest value in FP64. In FP32 the winner is
picked in FP32: a relative distance error e moves the closest point by up to
sqrt(2 e) d, 1e-3 d for e = 5e-7, on velocities that vary by about 1 per unit
length and d up to 3.5 cells: the wing test's 1e-3.
"""
import numpy as np
import pytest
import torch

from oracle import mask as OM
from paper_2002_08642_gb300 import build as pbuild
from paper_2002_08642_gb300 import inputs
from paper_2002_08642_gb300.solver import Solver

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    pbuild.build()


def _mesh(kind, dx):
    if kind == "small":      # one triangle below a cell, reach cut by the corner of the grid
        return np.array([[0.1, 0.1, 0.1], [0.3, 0.1, 0.1], [0.1, 0.25, 0.2]]) * dx, np.array([[0, 1, 2]])
    if kind == "outside":    # beyond a face: only part of the box lies in the grid
        return np.array([[1.9, 0.0, 0.0], [2.6, 0.1, 0.0], [2.0, 0.5, 0.3]]), np.array([[0, 1, 2]])
    if kind == "slivers":
        x = np.linspace(-0.8, 0.8, 9)
        xw = np.concatenate([np.stack([x, 0 * x, 0 * x], 1), np.stack([x, 0 * x + 1e-3 * dx, 0.2 * x], 1)])
        return xw, np.array([(i, i + 1, 9 + i) for i in range(8)] + [(i + 1, 9 + i, 10 + i) for i in range(8)])
    nc, ns = {"plate": (1, 1), "many": (41, 61)}[kind]   # 2 and 5002 triangles
    xw, _, tri, _ = inputs.plate(chord=0.6, span=1.4, nc=nc, ns=ns)
    return xw, tri


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("kind,n,half", [("small", 16, False), ("outside", 24, False), ("slivers", 32, False),
                                         ("plate", 32, True), ("plate", 48, False), ("many", 24, False)])
def test_rasterise_edges(kind, n, half, prec):
    L, nz = 4.0, n // 2 if half else n
    dx = L / n
    xw, tri = _mesh(kind, dx)
    tri = np.ascontiguousarray(tri, dtype=np.int32)
    om = np.array([0.3, -0.2, 0.9])
    vw = np.cross(om, xw)
    g = Solver(n, L, 1e-3, 1e-3, 5e-4, precision=prec, nz=nz)
    d = lambda a, t: torch.from_numpy(np.ascontiguousarray(a)).to("cuda", t)
    for call in range(2):
        O = (0.0, 0.0, 0.0) if kind == "small" else (2.0 + 0.1 * call, 2.0, 0.25 * nz * dx * (1 + call))
        fr = inputs.frame(inputs.rot_z(0.4 + call) @ inputs.rot_y(30.0), O, (0.1, 0.2, -0.1), (0.0, 0.1, 0.5))
        chi_o, us_o, _, _ = OM.rasterise(n, L, xw, vw, tri, fr, 2 * dx, 1.5 * dx, nz=nz)
        g.set_mask_from_nodes(d(xw, torch.float64), d(vw, torch.float64), d(tri, torch.int32), fr)
        chi, us = (f.double().cpu().numpy() for f in g.mask())
        assert chi_o.max() > 0
        assert np.abs(chi - chi_o).max() < (1e-12 if prec == "fp64" else 2e-6)
        both = (chi_o > 1e-9) & (chi > 1e-9)   # the rim's last cells may round to chi = 0 on one side
        du = np.abs(us - us_o)[:, both].max()
        print(kind, prec, "max chi error %.1e, max u_s error %.1e" % (np.abs(chi - chi_o).max(), du))
        assert du < (1e-12 * np.abs(us_o).max() if prec == "fp64" else 1e-3)
        assert np.all(us[:, chi == 0] == 0)
