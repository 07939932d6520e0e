"""Force and moment of FP32 contexts are sums in the precision of doubles.

The velocity is zero, so that the z pass's u is exactly 0 and q = -chi u_s of
given FP32 numbers: the reference sums the same q in rational arithmetic. dx,
eta and the moment point are dyadic, so that scaling is exact. Bound relative to
the sum S of the magnitudes of the terms: one rounding (u = 2^-53) of every
partial sum to a double, at most u S together, and the final double operations (dx
M + jo x F and the compensated pairs' last sums), at most 3 u S: 4 u S = 2^-51 S. A
sum of FP32 words of 48 bits is off by up to 2^-49 of a single term's moment, a
plain FP32 sum by 2^-25 or more. With u_s of both signs the terms cancel; the
moment point lies in the body or far outside the box.

With a flow the z pass rounds u itself; the last test compares an FP32 with an
FP64 context where the terms cancel.
"""
from fractions import Fraction

import numpy as np
import pytest
import torch

from paper_2002_08642_gb300 import build as pbuild
from paper_2002_08642_gb300.solver import Solver

pytestmark = pytest.mark.gpu

U51 = Fraction(1, 1 << 51)


@pytest.fixture(scope="module", autouse=True)
def _built():
    pbuild.build()


def _exact(n, pts, chi, us, x0, dx, scale):
    """(F, M) and the sums of their terms' magnitudes, as fractions."""
    F, M, aF, aM = ([Fraction(0)] * 3 for _ in range(4))
    for p, c, s in zip(pts, chi, us):
        q = [-Fraction(float(c)) * Fraction(float(v)) for v in s]
        r = [Fraction(int(i)) * dx - x for i, x in zip(p, x0)]
        for i in range(3):
            a, b = (i + 1) % 3, (i + 2) % 3
            F[i] += q[i]
            aF[i] += abs(q[i])
            M[i] += r[a] * q[b] - r[b] * q[a]
            aM[i] += abs(r[a] * q[b]) + abs(r[b] * q[a])
    return [f * scale for f in F + M], [f * scale for f in aF + aM]


def _forces(g, n, nz, pts, chi, us):
    i = tuple(torch.from_numpy(np.ascontiguousarray(pts[:, k])).cuda() for k in range(3))
    c = torch.zeros((n, n, nz), device="cuda")
    c[i] = torch.from_numpy(chi).cuda()
    s = torch.zeros((3, n, n, nz), device="cuda")
    s[(slice(None),) + i] = torch.from_numpy(np.ascontiguousarray(us.T)).cuda()
    g.set_velocity(torch.zeros((3, n, n, nz), device="cuda"))
    g.set_mask(c, s)
    g.step(1)
    F, M = g.forces()
    return list(F) + list(M)


# dx = 2^-4 or 2^-5; x0 in the box or far outside it (the offset then dominates)
@pytest.mark.parametrize("far", [False, True])
@pytest.mark.parametrize("n,nz", [(12, 12), (24, 24), (32, 16), (32, 32), (96, 96), (128, 64), (192, 192), (256, 256), (384, 384)])
def test_sums_are_as_exact_as_doubles(n, nz, far):
    dx, eta = Fraction(1, 32), Fraction(1, 512)
    x0 = [dx * v for v in ((-1000, 4000, 77777) if far else (n // 2, n // 3, nz // 2))]
    g = Solver(n, float(n * dx), 1e-3, float(eta), 1e-3, x0=[float(x) for x in x0], nz=nz)
    rng = np.random.default_rng(n + nz + far)
    f32 = lambda *a: rng.uniform(*a).astype(np.float32)  # noqa: E731
    worst = Fraction(0)
    for trial in range(30):
        if trial < 24:      # one point
            pts = np.stack([rng.integers(0, m, 1) for m in (n, n, nz)], 1)
        elif trial < 28:    # two whole lines and a scattered cloud, u_s of both signs
            y = int(rng.integers(0, n - 1))
            pts = np.concatenate([np.stack([np.full(nz, n // 2), np.full(nz, yy), np.arange(nz)], 1) for yy in (y, y + 1)] +
                                 [np.stack([rng.integers(0, m, 400) for m in (n, n, nz)], 1)])
            pts = np.unique(pts, axis=0)
        else:               # a block: every thread of some blocks has masked points
            s = [np.arange(m // 3, m // 3 + min(8, m // 3)) for m in (n, n, nz)]
            pts = np.stack(np.meshgrid(*s, indexing="ij"), -1).reshape(-1, 3)
        chi = f32(0.05, 1.0, len(pts))
        us = f32(-1.0, 1.0, (len(pts), 3)) * np.float32(10.0) ** rng.integers(-3, 3, (len(pts), 1)).astype(np.float32)
        us = us.astype(np.float32)
        got = _forces(g, n, nz, pts, chi, us)
        want, size = _exact(n, pts, chi, us, x0, dx, dx ** 3 / eta)
        for a, b, s in zip(got, want, size):
            worst = max(worst, abs(Fraction(a) - b) / s if s else abs(Fraction(a)))
    print(n, nz, far, "error / sum of magnitudes %.2f x 2^-53" % float(worst * (1 << 53)))
    assert worst <= U51
    g.close()


def test_cancellation_with_a_flow():
    """Points of one line whose q cancel to 1e-7 of their size, u of a smooth
    flow: the sum of FP32 q follows the FP64 context's to the rounding of u."""
    n, L = 64, 4.0
    z = np.arange(n)
    chi = np.zeros((n, n, n), dtype=np.float32)
    chi[20, 30], chi[20, 31] = 0.5, 0.5
    us = np.zeros((3, n, n, n), dtype=np.float32)
    big = (1000.0 * np.cos(2.0 * np.pi * z / n)).astype(np.float32)
    us[:, 20, 30], us[:, 20, 31] = big, -big
    x = 2.0 * np.pi * z / n
    u = np.zeros((3, n, n, n), dtype=np.float32)
    u[0] = np.sin(x)[:, None, None] * np.cos(x)[None, :, None]
    u[1] = -np.cos(x)[:, None, None] * np.sin(x)[None, :, None]
    out = {}
    for prec, dt in (("fp32", torch.float32), ("fp64", torch.float64)):
        g = Solver(n, L, 1e-3, 1e-3, 1e-4, precision=prec)
        g.set_velocity(torch.from_numpy(u).to("cuda", dt))
        g.set_mask(torch.from_numpy(chi).to("cuda", dt), torch.from_numpy(us).to("cuda", dt))
        g.step(1)
        out[prec] = np.array(g.forces()[0]) / ((L / n) ** 3 / 1e-3)
        g.close()
    # 128 points, chi = 1/2, u known to 20 roundings of 6e-8
    assert np.abs(out["fp32"] - out["fp64"]).max() < 128 * 0.5 * 20 * 6e-8
