"""The rasteriser with triangles that have no plane, each with nodes of its own
half a cell to two cells above a proper plate: two vertices at one place, all
three, and three on a line (whose cross product is rounding). Such a
triangle takes no points of the mask away: chi is at least the plate's own
(1e-12 in FP64; the FP32 walk's winner may be farther by a relative 5e-7, 2e-6
in chi as for the wing). With coincident vertices it is a segment or a point,
and chi that of the least distance to the plate and to those.
"""
import numpy as np
import pytest
import torch

from oracle import mask as OM
from paper_2002_08642_gb300 import build as pbuild
from paper_2002_08642_gb300 import inputs
from paper_2002_08642_gb300.solver import Solver

pytestmark = pytest.mark.gpu

N, L = 32, 4.0
DX = L / N
TOL = {"fp64": 1e-12, "fp32": 2e-6}


@pytest.fixture(scope="module", autouse=True)
def _built():
    pbuild.build()


def _extra(kind, at, rng):
    """Nodes of one triangle near `at` that has no area."""
    d = rng.standard_normal(3)
    d *= 2.0 * DX / np.linalg.norm(d)
    if kind == "ab":
        return np.stack([at, at, at + d])
    if kind == "ac":
        return np.stack([at, at + d, at])
    if kind == "bc":
        return np.stack([at + d, at, at])
    if kind == "abc":
        return np.stack([at, at, at])
    return np.stack([at, at + rng.uniform(0.2, 0.8) * d, at + d])   # on a line, up to rounding


def _rasterise(xw, tri, prec, fr):
    d = lambda a, t: torch.from_numpy(np.ascontiguousarray(a)).to("cuda", t)
    g = Solver(N, L, 1e-3, 1e-3, 5e-4, precision=prec)
    g.set_mask_from_nodes(d(xw, torch.float64), d(np.zeros_like(xw), torch.float64), d(tri, torch.int32), fr)
    chi = g.mask()[0].double().cpu().numpy()
    g.close()
    return chi


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("kind", ["ab", "ac", "bc", "abc", "line"])
def test_triangles_without_a_plane_take_no_points(kind, prec):
    rng = np.random.default_rng(len(kind) + ord(kind[0]))
    xw, _, tri, _ = inputs.plate(chord=0.8, span=1.2, nc=4, ns=6)
    fr = inputs.frame(inputs.rot_z(0.4) @ inputs.rot_y(30.0), (2.0, 2.03, 1.98))
    chi_o = OM.rasterise(N, L, xw, np.zeros_like(xw), tri, fr, 2 * DX, 1.5 * DX)[0]
    lo, hi = xw.min(0), xw.max(0)
    normal = np.cross(xw[tri[0, 1]] - xw[tri[0, 0]], xw[tri[0, 2]] - xw[tri[0, 0]])
    normal /= np.linalg.norm(normal)
    nodes, tris = [xw], [tri]
    for k in range(24):
        at = lo + (hi - lo) * rng.uniform(0.1, 0.9, 3) + rng.uniform(0.5, 2.0) * DX * normal
        tris.append(np.arange(3)[None] + sum(len(q) for q in nodes))
        nodes.append(_extra(kind, at, rng))
    xe, te = np.concatenate(nodes), np.concatenate(tris).astype(np.int32)
    chi = _rasterise(xe, te, prec, fr)
    worst = (chi_o - chi).max()
    print(kind, prec, "largest chi lost %.1e" % worst)
    assert worst < TOL[prec]
    assert chi.max() <= 1.0
    if kind != "line":
        d = OM.rasterise(N, L, xw, np.zeros_like(xw), tri, fr, 2 * DX, 1.5 * DX)[3]
        xg = OM.global_nodes(xe, fr)
        X = np.stack(np.meshgrid(*[np.arange(N) * DX] * 3, indexing="ij"), -1)
        for t in te[len(tri):]:
            a, e = xg[t[0]], max((xg[t[1]] - xg[t[0]], xg[t[2]] - xg[t[0]]), key=lambda q: q @ q)
            q = np.clip(((X - a) @ e) / max(e @ e, 1e-300), 0.0, 1.0)
            d = np.minimum(d, np.linalg.norm(X - a - q[..., None] * e, axis=-1))
        assert np.abs(chi - OM.chi_cos(d, 2 * DX, 1.5 * DX)).max() < TOL[prec]
