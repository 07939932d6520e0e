"""Line lengths at the edges of the transforms' plans (n = 2^a and 3 2^a,
radix 4 and 16, one to three stages, padded and unpadded sub-lines, batches
that end in partial warps), cubic and n x n x n/2, for the passes that choose
by length: the step with forces, the step with the sponge, the reversed step.

FP64 against the oracle at the small sizes: the tolerances of the step and
adjoint tests (1e-12 per step, 1e-10). FP32 against the FP64 path at the
larger ones: rounding of about 3 log2(n) stages of u = 6e-8 each in a
transform, forward and inverse, a random walk of about 7 u per pass and three
passes: below 2e-6 relative in the L2 norm for velocity and gradients. That
holds for dJ/dchi only while no complex line carries two vectors of unlike
size.
"""
import numpy as np
import pytest
import torch

from oracle import adjoint as OA
from oracle import step as S
from paper_2002_08642_gb300 import build as pbuild
from paper_2002_08642_gb300 import inputs
from paper_2002_08642_gb300.solver import Solver

pytestmark = pytest.mark.gpu

L, NU, ETA, DT = 4.0, 0.02, 0.05, 2e-3
A, B = np.array([0.3, -0.2, 1.0]), np.array([0.1, 0.4, -0.3])


@pytest.fixture(scope="module", autouse=True)
def _built():
    pbuild.build()


def rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


def _fields(n, nz, steps):
    """Seeded velocity, masks on a block that ends inside a line, solid velocities, sponge."""
    rng = np.random.default_rng(n + nz)
    u = inputs.random_field(n, L, seed=n + 5, rms=0.3, nz=nz)
    masks = []
    for _ in range(steps):
        chi = np.zeros((n, n, nz))
        sl = (slice(n // 4, n // 4 + n // 3), slice(n // 3, n // 3 + n // 4 + 1), slice(nz // 5, nz // 5 + nz // 2))
        chi[sl] = rng.uniform(0.2, 1.0, chi[sl].shape)
        masks.append((chi, rng.standard_normal((3, n, n, nz)) * 0.1))
    sp = np.zeros((n, n, nz))
    sp[: n // 8 + 1] = 1.0
    return u, masks, sp


def _run(n, nz, prec, u, masks, sp, adjoint):
    dt = torch.float64 if prec == "fp64" else torch.float32
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda", dt)
    g = Solver(n, L, NU, ETA, DT, precision=prec, x0=(1.9, 2.1, 0.9), nz=nz, with_adjoint=adjoint)
    g.set_velocity(d(u))
    if sp is not None:
        g.set_sponge(d(sp), 0.3)
    states, fm = [], []
    for chi, us in masks:
        if adjoint:
            states.append(g.state_buffer())
            g.save_state(states[-1])
        g.set_mask(d(chi), d(us))
        g.step(1)
        F, M = g.forces()
        fm.append(list(F) + list(M))
    out = {"u": g.velocity().double().cpu().numpy(), "fm": np.array(fm)}
    if adjoint:
        gchi = torch.empty((n, n, nz), dtype=dt, device="cuda")
        gus = torch.empty((3, n, n, nz), dtype=dt, device="cuda")
        g.adjoint_reset()
        for k in range(len(masks) - 1, -1, -1):
            g.restore_state(states[k])
            g.set_mask(*(d(f) for f in masks[k]))
            g.adjoint_step(A / len(masks), B / len(masks), k == 0, gchi, gus)
        out["chi"], out["us"] = gchi.double().cpu().numpy(), gus.double().cpu().numpy()
    g.close()
    return out


@pytest.mark.parametrize("n,nz,sponge", [(12, 12, False), (12, 12, True), (16, 16, False), (24, 24, True), (32, 16, False),
                                         (48, 24, True), (48, 48, False), (64, 32, False)])
def test_fp64_against_oracle(n, nz, sponge):
    u, masks, sp = _fields(n, nz, 2)
    o = S.Solver(S.Params(n=n, L=L, nu=NU, eta=ETA, dt=DT, x0=(1.9, 2.1, 0.9), nz=nz))
    o.set_velocity(u)
    if sponge:
        o.set_sponge(sp, 0.3)
    fm = []
    for chi, us in masks:
        o.set_mask(chi, us)
        o.step(1)
        fm.append(list(o.F) + list(o.M))
    got = _run(n, nz, "fp64", u, masks, sp if sponge else None, False)
    assert rel(got["u"], o.velocity()) < 2e-12
    assert rel(got["fm"], np.array(fm)) < 1e-12


@pytest.mark.parametrize("n,nz", [(12, 12), (32, 32), (32, 16), (48, 48)])
def test_fp64_adjoint_against_oracle(n, nz):
    u, masks, _ = _fields(n, nz, 2)
    p = S.Params(n=n, L=L, nu=NU, eta=ETA, dt=DT, x0=(1.9, 2.1, 0.9), nz=nz)
    _, states = OA.forward(p, u, masks, np.full(2, 0.5), A, B)
    gchi, gus = OA.adjoint(p, states, masks, np.full(2, 0.5), A, B)
    got = _run(n, nz, "fp64", u, masks, None, True)
    assert rel(got["chi"], gchi[0]) < 1e-10 and rel(got["us"], gus[0]) < 1e-10


@pytest.mark.parametrize("n,nz,sponge", [(48, 48, False), (64, 64, True), (96, 96, False), (96, 48, True), (128, 128, False),
                                         (192, 96, True), (192, 192, False), (256, 128, False)])
def test_fp32_against_fp64(n, nz, sponge):
    u, masks, sp = _fields(n, nz, 2)
    u, masks = u.astype(np.float32), [(c.astype(np.float32), s.astype(np.float32)) for c, s in masks]
    got = {q: _run(n, nz, q, u, masks, sp if sponge else None, not sponge) for q in ("fp32", "fp64")}
    err = {k: rel(got["fp32"][k], got["fp64"][k]) for k in got["fp32"]}
    print(n, nz, {k: "%.1e" % v for k, v in err.items()})
    assert err["u"] < 2e-6 and err["fm"] < 2e-6
    assert err.get("chi", 0.0) < 2e-6 and err.get("us", 0.0) < 2e-6
