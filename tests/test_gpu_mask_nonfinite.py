"""Nodes that are no numbers (a coupled run that diverged, a bad input): their
triangles leave the mask alone and cost nothing. chi and u_s are those of the
mesh without them, bit for bit, in both precisions; a mesh of NaN nodes only
gives an empty mask in well under the time of a walk over the grid (2000
triangles x 256^3 points would be 3e10 pair tests, 50 ms and more; the call takes
about 0.1 ms).
"""
import numpy as np
import pytest
import torch

from paper_2002_08642_gb300 import build as pbuild
from paper_2002_08642_gb300 import inputs
from paper_2002_08642_gb300.solver import Solver

pytestmark = pytest.mark.gpu

L = 4.0
d = lambda a, t: torch.from_numpy(np.ascontiguousarray(a)).to("cuda", t)  # noqa: E731


@pytest.fixture(scope="module", autouse=True)
def _built():
    pbuild.build()


def _rasterise(g, xw, tri, fr):
    vw = np.cross([0.3, -0.2, 0.9], np.where(np.isfinite(xw), xw, 0.0))
    g.set_mask_from_nodes(d(xw, torch.float64), d(vw, torch.float64), d(tri, torch.int32), fr)
    return [f.cpu().numpy() for f in g.mask()]


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("bad", [np.nan, -np.nan, np.inf, -np.inf])
def test_triangles_of_nonfinite_nodes_are_left_out(bad, prec):
    n = 32
    xw, _, tri, _ = inputs.plate(chord=0.8, span=1.2, nc=4, ns=6)
    fr = inputs.frame(inputs.rot_z(0.4) @ inputs.rot_y(30.0), (2.0, 2.03, 1.98))
    k = len(xw)
    extra = np.stack([[bad, 0.1, 0.2], [0.1, bad, 0.2], [bad, bad, bad], [bad, 0.0, bad], [0.2, 0.1, bad]])
    more = [(k, 0, 5), (3, k + 1, 7), (1, 6, k + 2), (k + 2, k + 2, k + 2), (k, k + 1, k + 4), (k + 3, 4, k + 2)]
    g = Solver(n, L, 1e-3, 1e-3, 5e-4, precision=prec)
    want = _rasterise(g, xw, tri, fr)
    assert want[0].max() == 1.0
    got = _rasterise(g, np.concatenate([xw, extra]), np.concatenate([more[:3], tri, more[3:]]).astype(np.int32), fr)
    assert np.array_equal(got[0], want[0]) and np.array_equal(got[1], want[1])
    g.close()


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_a_mesh_of_nan_nodes_costs_nothing(prec):
    g = Solver(256, L, 1e-3, 1e-3, 5e-4, precision=prec)
    xw = d(np.full((1002, 3), np.nan), torch.float64)
    i = np.arange(2000)
    tri = d(np.stack([i % 1000, (i + 1) % 1000, (i + 2) % 1000], 1), torch.int32)
    fr = inputs.frame(np.eye(3), (2.0, 2.0, 2.0))
    e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    g.set_mask_from_nodes(xw, xw, tri, fr)
    e0.record()
    g.set_mask_from_nodes(xw, xw, tri, fr)
    e1.record()
    torch.cuda.synchronize()
    assert e0.elapsed_time(e1) < 5.0
    chi, us = g.mask()
    assert not chi.any() and not us.any()
    g.close()
