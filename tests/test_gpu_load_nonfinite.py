"""Nodes that are no numbers have no grid points around them: their pressure is
0 (as every weight beyond 2.5 cells is), and the other nodes' pressures and loads
are those of the same mesh without them, bit for bit."""
import numpy as np
import pytest
import torch

from paper_2002_08642_gb300 import build as pbuild
from paper_2002_08642_gb300 import inputs
from paper_2002_08642_gb300.solver import Solver

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    pbuild.build()


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_nonfinite_nodes(bad, prec):
    n, L = 24, 4.0
    dt = torch.float64 if prec == "fp64" else torch.float32
    xw, tri = inputs.elliptic_wing_mesh(60)
    k = len(xw)
    xb = np.concatenate([xw, [[bad, 0.1, 0.2], [bad, bad, bad]]])
    tb = np.concatenate([tri, [[k, k + 1, k]]]).astype(np.int32)   # a triangle of their own
    fr = inputs.frame(np.eye(3), (2.0, 2.0, 2.0))
    g = Solver(n, L, 1e-3, 1e-3, 5e-4, precision=prec)
    p = torch.from_numpy(np.random.default_rng(1).standard_normal((n, n, n))).to("cuda", dt)
    d = lambda a, t: torch.from_numpy(np.ascontiguousarray(a)).to("cuda", t)  # noqa: E731
    pn, fn = g.pressure_loads(p, d(xw, torch.float64), d(tri, torch.int32), fr)
    pb, fb = g.pressure_loads(p, d(xb, torch.float64), d(tb, torch.int32), fr)
    assert torch.equal(pb[:k], pn) and torch.equal(fb[:k], fn)
    assert torch.equal(pb[k:], torch.zeros(2, dtype=torch.float64, device="cuda"))
    g.close()
