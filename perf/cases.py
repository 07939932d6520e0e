"""Performance cases of the penalized pseudo-spectral solver: the work that a
program using this package has it do, each pass through the public entry
points (``Solver``, ``FSI``, ``TimeAveragedForce``).

A case is a dict of plain values:

* ``kind``  what one pass does (see ``run``);
* ``n``, ``half``  grid n x n x n, or n x n x n/2 (the 4 x 4 x 2 box) if half;
* ``fp64``  precision of the solver (FP32 transforms otherwise);
* ``nodes``  mesh nodes of the wing (0: no wing; the flat plate's two
  triangles are fixed by its kind); ``steps``  time steps of a pass;
* ``sponge``  the vorticity-damping term on.

Numbers that a solver of FP32 fields gives in 64-bit containers (forces, node
loads, node positions) come back as 32-bit values: that is the accuracy of
the fields they are sums of. The FP64 cases return them as they are.

``exact`` is a plain torch evaluation in 64 bits of the same equations; the
package's ``inputs`` module, which holds input recipes only and none of the
solver's arithmetic, makes the meshes and motions for both.
"""
import math

import numpy as np
import torch

from paper_2002_08642_gb300 import inputs

# the revolving-wing runs: box, viscosity (Re = 1800 on the span), penalization, step
L, NU, ETA, DT = 4.0, 1.527e-4, 1e-3, 5e-4
# the decaying periodic flow of the solver's first validation run
DECAY = dict(L=2.0 * math.pi, nu=0.01, eta=1.0, dt=1e-3)
C_SP = 0.05           # sponge constant of the damped outer shell
POSITIONS = 8         # wing positions a program has ahead of it; a pass uses the next ones
EVERY = 4             # checkpoint interval of a gradient window
SIZES = (12, 16, 24, 32, 48, 64, 96, 128, 192, 256, 384, 512, 768)


def _case(kind, n, fp64=False, nodes=0, steps=1, half=False, sponge=False):
    return {"kind": kind, "n": n, "half": half, "fp64": fp64, "nodes": nodes, "steps": steps, "sponge": sponge}


def listed():
    return [
        # the smallest run: a decaying periodic box, all its steps from one call; launches and latency
        dict(_case("decay", 32, fp64=True, steps=20), name="decay_32_fp64"),
        # a coarse wing run as used to set up a study: small mesh, force read back every step
        dict(_case("wing", 48, nodes=121, steps=8), name="wing_48"),
        # static plate in a random flow, steps without a host in between (the 128^3 configuration)
        dict(_case("plate", 128, steps=10), name="plate_128"),
        # FP64 reference run that an FP32 run is compared with
        dict(_case("wing", 128, fp64=True, nodes=600, steps=2), name="wing_128_fp64"),
        # the 256^3 flexible-wing configuration: mask rasterised and force read every step
        dict(_case("wing", 256, nodes=600, steps=4), name="wing_256"),
        # the paper's 4 x 4 x 2 box, sponge on, n = 3M lines
        dict(_case("wing", 384, nodes=1065, steps=2, half=True, sponge=True), name="box_384_sponge"),
        # the production size: 768^3, 2000 nodes
        dict(_case("wing", 768, nodes=2000, steps=2), name="wing_768"),
        # a new initial field and a velocity snapshot (restart from a file, output)
        dict(_case("fields", 384), name="fields_384"),
        # pressure snapshot and the loads on the wing
        dict(_case("pressure", 192, nodes=833), name="pressure_192"),
        # coupled fluid-structure step, 48 x 16 vein/membrane network on the host
        dict(_case("fsi", 256, nodes=833), name="fsi_256"),
        # two reversed steps of a checkpointed window (backward alone): the gradients with respect to the
        # mask and the solid velocity. Their sum into the mesh nodes cancels a thousandfold between the
        # wing's two sides (2e-4 off in FP32); it is compared in the FP64 window below
        dict(_case("adjoint", 512, nodes=600, steps=2), name="adjoint_512"),
        # a whole gradient of the mean lift: forward window, recompute, reversal (forward and backward)
        dict(_case("gradient", 64, fp64=True, nodes=157, steps=8), name="gradient_64_fp64"),
    ]


def draw(rng):
    """One more case. Grid sizes are those the library is built for, node and
    step counts spread over the logarithm of their ranges, odd ones included."""
    def size(lo, hi):
        return rng.choice([s for s in SIZES if lo <= s <= hi])

    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["decay", "wing", "wing", "wing", "plate", "fields", "pressure", "fsi", "adjoint", "gradient"])
    if kind == "decay":
        return _case(kind, size(12, 96), fp64=rng.random() < 0.5, steps=log(5, 40))
    if kind == "plate":
        return _case(kind, size(48, 192), fp64=rng.random() < 0.2, steps=log(2, 20))
    if kind == "wing":
        fp64 = rng.random() < 0.2
        n = size(32, 128) if fp64 else size(32, 512)
        return _case(kind, n, fp64=fp64, nodes=log(60, 2000), steps=log(1, 6),
                     half=n >= 64 and rng.random() < 0.3, sponge=rng.random() < 0.25)
    if kind == "fields":
        return _case(kind, size(16, 512), fp64=rng.random() < 0.2, half=False)
    if kind == "pressure":
        n = size(32, 384)
        return _case(kind, n, nodes=log(60, 2000), half=n >= 64 and rng.random() < 0.3)
    if kind == "fsi":
        ns = rng.randint(12, 48)
        return _case(kind, size(48, 256), nodes=(ns + 1) * (8 * (1 + (ns > 30)) + 1))
    if kind == "adjoint":
        return _case(kind, size(48, 384), fp64=False, nodes=log(60, 1200), steps=2)
    return _case(kind, size(24, 64), fp64=True, nodes=log(60, 600), steps=log(3, 9))


# ------------------------------------------------------------------- inputs
def _nz(case):
    return case["n"] // 2 if case["half"] else case["n"]


def _params(case):
    if case["kind"] == "decay":
        return DECAY
    return dict(L=L, nu=NU, eta=ETA, dt=DT)


def _dtype(case):
    return torch.float64 if case["fp64"] else torch.float32


def _velocity(case, seed):
    """Random field with a k^(-5/3) spectrum, 1 <= |m| < n/3, rms about 0.05
    per component; the decaying flow adds it to the 3-D Taylor-Green vortex."""
    n, nz, dt = case["n"], _nz(case), _dtype(case)
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    m = torch.fft.fftfreq(n, 1.0 / n, device="cuda", dtype=dt)
    mz = torch.arange(nz // 2 + 1, device="cuda", dtype=dt) * (n / nz)
    k2 = m[:, None, None] ** 2 + m[None, :, None] ** 2 + mz[None, None, :] ** 2
    band = (k2 >= 1.0) & (k2 < (n / 3.0) ** 2)
    amp = torch.where(band, torch.where(band, k2, torch.ones_like(k2)).pow(-11.0 / 12.0), torch.zeros_like(k2))
    del k2, band
    u = torch.empty((3, n, n, nz), dtype=dt, device="cuda")
    for c in range(3):
        f = torch.fft.rfftn(torch.randn((n, n, nz), generator=g, dtype=dt, device="cuda"))
        u[c] = torch.fft.irfftn(f * amp, s=(n, n, nz))
        del f
        u[c] *= 0.05 * math.sqrt(1.5) / u[c].double().square().mean().sqrt().item()
    if case["kind"] == "decay":
        x = torch.arange(n, device="cuda", dtype=dt) * (2.0 * math.pi / n)
        X, Y, Z = x[:, None, None], x[None, :, None], x[None, None, :]
        u[0] += torch.sin(X) * torch.cos(Y) * torch.cos(Z)
        u[1] -= torch.cos(X) * torch.sin(Y) * torch.cos(Z)
    return u


def _mesh(case):
    return inputs.elliptic_wing_mesh(case["nodes"])


def _centre(case):
    return (0.5 * L, 0.5 * L, 0.5 * L * _nz(case) / case["n"])


def _motion(case, seed, count):
    """`count` successive positions of the revolving, flapping wing from a
    seeded time on: (triangles, rest nodes, [(nodes, velocities, frame)])."""
    xw0, tri = _mesh(case)
    amp = inputs.flapping_amplitudes(xw0, seed=int(seed) % (1 << 31))
    t0 = np.random.default_rng(int(seed)).uniform(0.0, 1.0)
    return tri, xw0, [inputs.revolving_wing(t0 + k * DT, xw0, amp, centre=_centre(case)) for k in range(count)]


def _plate():
    """Chord 0.3, span 1, two triangles, 30 degrees, centred in the box."""
    return inputs.plate()


def _fsi_wing(case):
    nc = 16 if case["nodes"] % 17 == 0 else 8
    return inputs.fsi_wing(ns=case["nodes"] // (nc + 1) - 1, nc=nc, veins=tuple(range(0, nc + 1, 4)))


def _frames(t):
    return inputs.revolving_frames(t, tau=0.4)


def _sponge(case):
    """Damping in the outer 1/16 of the box along x and y."""
    n, nz = case["n"], _nz(case)
    i = torch.arange(n, device="cuda")
    edge = ((i < n // 16) | (i >= n - n // 16)).to(_dtype(case))
    return torch.maximum(edge[:, None, None], edge[None, :, None]).expand(n, n, nz).contiguous()


def _gpu(a, dt=torch.float64):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda", dt)


# ---------------------------------------------------------- prepare and run
def prepare(case, seed):
    from paper_2002_08642_gb300.solver import Solver

    kind, n, nz = case["kind"], case["n"], _nz(case)
    p = _params(case)
    g = Solver(n, p["L"], p["nu"], p["eta"], p["dt"], precision="fp64" if case["fp64"] else "fp32", nz=nz,
               mask_profile="tanh" if kind == "plate" else "cos", with_adjoint=kind in ("adjoint", "gradient"),
               keep_uw=kind == "fsi")
    u = _velocity(case, seed)
    s = {"kind": kind, "solver": g, "steps": case["steps"], "fp64": case["fp64"]}
    if kind == "fields":
        s["u"] = u
        s["out"] = torch.empty_like(u)
        return s
    g.set_velocity(u)
    if kind in ("decay", "plate", "wing"):
        s["out"] = torch.empty_like(u)
    if kind == "plate":
        xw, vw, tri, fr = _plate()
        g.set_mask_from_nodes(_gpu(xw), _gpu(vw), _gpu(tri, torch.int32), fr)
    if kind in ("wing", "pressure", "adjoint", "gradient"):
        tri, xw0, seq = _motion(case, seed, POSITIONS + 1)
        s["tri"] = _gpu(tri, torch.int32)
        s["x"] = [_gpu(q[0]) for q in seq]
        s["v"] = [_gpu(q[1]) for q in seq]
        s["frame"] = [q[2] for q in seq]
    if kind == "wing":
        s["at"] = 0
        if case["sponge"]:
            g.set_sponge(_sponge(case), C_SP)
    if kind == "pressure":
        g.set_mask_from_nodes(s["x"][0], s["v"][0], s["tri"], s["frame"][0])
        g.step(2)
        s["p"] = torch.empty((n, n, nz), dtype=_dtype(case), device="cuda")
    if kind == "fsi":
        from paper_2002_08642_gb300.fsi import FSI
        from paper_2002_08642_gb300.massspring import MassSpring

        w = _fsi_wing(case)
        ms = MassSpring(w["x0"], w["mass"], w["ext"], w["ke"], w["bend"], w["kb"], fixed=w["fixed"])
        s["fsi"] = FSI(g, ms, w["tri"], _frames)
    if kind == "adjoint":
        # forward states before the two steps to be reversed, as a window's recompute leaves them
        s["states"] = []
        for k in range(2):
            g.set_mask_from_nodes(s["x"][k], s["v"][k], s["tri"], s["frame"][k])
            g.step(1)
            s["states"].append(g.state_buffer())
            g.save_state(s["states"][k])
        s["gchi"] = [torch.empty((n, n, nz), dtype=_dtype(case), device="cuda") for k in range(2)]
        s["gus"] = [torch.empty((3, n, n, nz), dtype=_dtype(case), device="cuda") for k in range(2)]
    if kind == "gradient":
        from paper_2002_08642_gb300.adjoint import WingWindow

        steps = case["steps"]
        s["xw0"] = _gpu(xw0)
        pos = [k % POSITIONS for k in range(steps)]
        s["window"] = WingWindow(s["tri"], [s["x"][k] - s["xw0"] for k in pos], [s["v"][k] for k in pos],
                                 [s["frame"][k] for k in pos], u)
    return s


ADJ_F, ADJ_M = (0.0, 0.2, 0.5), (0.1, 0.0, -0.3)   # weights of force and moment in the reversed steps


def _as(s, values):
    return np.asarray(values, dtype=np.float64 if s["fp64"] else np.float32)


def run(s):
    g, kind = s["solver"], s["kind"]
    if kind == "decay":
        g.step(s["steps"])
        return g.velocity(out=s["out"])
    if kind == "plate":
        g.step(s["steps"])
        F, M = g.forces()
        return {"force": _as(s, list(F) + list(M)), "u": g.velocity(out=s["out"])}
    if kind == "wing":
        fm = []
        for _ in range(s["steps"]):
            k = s["at"] % POSITIONS
            s["at"] += 1
            g.set_mask_from_nodes(s["x"][k], s["v"][k], s["tri"], s["frame"][k])
            g.step(1)
            F, M = g.forces()
            fm.append(list(F) + list(M))
        return {"force": _as(s, fm), "u": g.velocity(out=s["out"])}
    if kind == "fields":
        g.set_velocity(s["u"])
        return g.velocity(out=s["out"])
    if kind == "pressure":
        g.pressure(out=s["p"])
        pn, fn = g.pressure_loads(s["p"], s["x"][0], s["tri"], s["frame"][0])
        return {"p": s["p"], "p_nodes": pn.to(s["p"].dtype), "f_nodes": fn.to(s["p"].dtype)}
    if kind == "fsi":
        s["fsi"].step(1)
        x, v = s["fsi"].state()
        return {"p": s["fsi"].p, "f": _as(s, s["fsi"].f_wing), "x": _as(s, x), "v": _as(s, v)}
    if kind == "adjoint":
        g.adjoint_reset()
        for k in (1, 0):
            g.restore_state(s["states"][k])
            g.set_mask_from_nodes(s["x"][k + 1], s["v"][k + 1], s["tri"], s["frame"][k + 1])
            g.adjoint_step(ADJ_F, ADJ_M, False, s["gchi"][k], s["gus"][k])
        return {"chi": s["gchi"], "us": s["gus"]}
    from paper_2002_08642_gb300.adjoint import TimeAveragedForce

    xw = s["xw0"].clone().requires_grad_(True)
    J = TimeAveragedForce.apply(xw, g, s["window"], EVERY)
    J[2].backward()
    return {"mean": J.detach(), "xw": xw.grad}


# -------------------------------------------------------------------- work
def work(case):
    """Bytes: the inputs of a pass read once and its outputs written once (the
    two kept spectral states of a step, the fields given and returned).
    Flops: the line transforms of the kept modes, 5 m log2 m each, and the
    pointwise terms."""
    n, nz, steps, kind = case["n"], _nz(case), case["steps"], case["kind"]
    e = 8 if case["fp64"] else 4
    K, Kz = 2 * ((n - 1) // 3) + 1, (nz - 1) // 3 + 1
    pts, state = n * n * nz, 2 * 3 * K * K * Kz * 2 * e

    def fft(fields):   # 3-D transforms of real fields: x lines, y lines, z lines (two fields each)
        line = lambda m: 5.0 * m * math.log2(m)  # noqa: E731
        return fields * (K * Kz * line(n) + n * Kz * line(n) + 0.5 * n * n * line(nz))

    step_b, step_f = 2 * state, fft(12 if case["sponge"] else 9) + 40.0 * pts
    if case["sponge"]:
        step_b += pts * e
    mesh = 72 * case["nodes"] * steps
    out = 3 * pts * e
    if kind in ("decay", "wing"):
        # the states between the steps of one pass need not leave the chip
        return {"bytes": step_b + out + mesh, "flops": steps * step_f + fft(3)}
    if kind == "plate":
        return {"bytes": step_b + out + 4 * pts * e, "flops": steps * step_f + fft(3)}
    if kind == "fields":
        return {"bytes": 2 * out + state, "flops": fft(6) + 15.0 * pts}
    if kind == "pressure":
        return {"bytes": state // 2 + pts * e + mesh, "flops": fft(10) + 40.0 * pts}
    if kind == "fsi":
        return {"bytes": step_b + pts * e + mesh, "flops": step_f + fft(4) + 20.0 * pts}
    rev = fft(15) + 120.0 * pts
    if kind == "adjoint":
        # per reversed step the forward state, the adjoint state updated, both gradients written
        return {"bytes": steps * (state + 2 * state + 4 * pts * e), "flops": steps * rev}
    return {"bytes": 2 * state + out + 2 * mesh, "flops": 2 * steps * step_f + steps * rev}


# ------------------------------------------------------------------- exact
class _Exact:
    """The equations in 64 bits with torch's transforms, full half spectra."""

    def __init__(self, case):
        p = _params(case)
        self.n, self.nz, self.eta, self.dt = case["n"], _nz(case), p["eta"], p["dt"]
        self.dx, self.L = p["L"] / case["n"], p["L"]
        n, nz, f8 = self.n, self.nz, dict(device="cuda", dtype=torch.float64)
        m = torch.fft.fftfreq(n, 1.0 / n, **f8)
        mz = torch.arange(nz // 2 + 1, **f8)
        kx = 2.0 * math.pi / p["L"] * m
        kz = 2.0 * math.pi / (p["L"] * nz / n) * mz
        self.k = (kx[:, None, None], kx[None, :, None], kz[None, None, :])
        self.keep = ((3 * m.abs() < n)[:, None, None] & (3 * m.abs() < n)[None, :, None] & (3 * mz < nz)[None, None, :])
        ex, ez = torch.exp(-p["nu"] * kx * kx * p["dt"]), torch.exp(-p["nu"] * kz * kz * p["dt"])
        self.E = ex[:, None, None] * ex[None, :, None] * ez[None, None, :]
        self.chi_sp = _sponge(case).double() if case["sponge"] else None
        c = [0.5 * p["L"]] * 2 + [0.5 * p["L"] * nz / n]
        self.r = [(torch.arange(q, **f8) * self.dx - c[a]) for a, q in enumerate((n, n, nz))]

    def fwd(self, f):
        return torch.fft.rfftn(f) * self.keep

    def inv(self, f):
        return torch.fft.irfftn(f, s=(self.n, self.n, self.nz))

    def k2(self):
        k2 = self.k[0] ** 2 + self.k[1] ** 2 + self.k[2] ** 2
        k2[0, 0, 0] = 1.0
        return k2

    def project(self, f, mean):
        d = (self.k[0] * f[0] + self.k[1] * f[1] + self.k[2] * f[2]) / self.k2()
        out = [f[c] - self.k[c] * d for c in range(3)]
        if not mean:
            zero = torch.ones((self.n, self.n, self.nz // 2 + 1), device="cuda", dtype=torch.float64)
            zero[0, 0, 0] = 0.0
            out = [o * zero for o in out]
        return out

    def velocity_hat(self, u):
        return self.project([self.fwd(u[c].double()) for c in range(3)], True)

    def cross_k(self, f, c):
        a, b = (c + 1) % 3, (c + 2) % 3
        return 1j * (self.k[a] * f[b] - self.k[b] * f[a])

    def rhs(self, uh, chi, us):
        """(N_hat before the projection, physical u)."""
        w = [self.inv(self.cross_k(uh, c)) for c in range(3)]
        u = [self.inv(uh[c]) for c in range(3)]
        sp = None
        if self.chi_sp is not None:
            sh = [self.fwd(self.chi_sp * w[c]) for c in range(3)]
            sp = [-self.cross_k(sh, c) / (C_SP * self.k2()) for c in range(3)]
        N = []
        for c in range(3):
            a, b = (c + 1) % 3, (c + 2) % 3
            q = u[a] * w[b] - u[b] * w[a]
            if chi is not None:
                q = q - chi / self.eta * (u[c] - us[c])
            N.append(self.fwd(q))
            if sp is not None:
                N[c] = N[c] + sp[c]
        return N, u

    def force(self, u, chi, us):
        q = [chi * (u[c] - us[c]) for c in range(3)]
        x, y, z = self.r[0][:, None, None], self.r[1][None, :, None], self.r[2][None, None, :]
        m = [y * q[2] - z * q[1], z * q[0] - x * q[2], x * q[1] - y * q[0]]
        return torch.stack([f.sum() for f in q + m]) * self.dx ** 3 / self.eta

    def step(self, uh, prev, chi, us):
        """(u_hat^{n+1}, P N_hat^n, forces of u^n); prev None: the Euler start."""
        N, u = self.rhs(uh, chi, us)
        fm = self.force(u, chi, us) if chi is not None else None
        del u
        N = self.project(N, False)
        if prev is None:
            new = [self.E * (uh[c] + self.dt * N[c]) for c in range(3)]
        else:
            new = [self.E * uh[c] + 0.5 * self.dt * (3.0 * self.E * N[c] - self.E * self.E * prev[c]) for c in range(3)]
        return new, N, fm

    def pressure(self, uh, chi, us):
        N, u = self.rhs(uh, chi, us)
        ph = -1j * (self.k[0] * N[0] + self.k[1] * N[1] + self.k[2] * N[2]) / self.k2()
        ph[0, 0, 0] = 0.0
        return self.inv(ph) - 0.5 * (u[0] ** 2 + u[1] ** 2 + u[2] ** 2)

    # ------------------------------------------------ mask from triangles
    @staticmethod
    def closest(P, X):
        """Barycentric weights of the closest point of triangle X (m, 3 vertices, 3) to P (m, 3):
        the plane projection where it falls inside, else the nearest point of the three edges."""
        a = X[:, 0]
        e0, e1, d = X[:, 1] - a, X[:, 2] - a, P - a
        m00, m01, m11 = (e0 * e0).sum(1), (e0 * e1).sum(1), (e1 * e1).sum(1)
        r0, r1 = (e0 * d).sum(1), (e1 * d).sum(1)
        det = m00 * m11 - m01 * m01
        s, t = (m11 * r0 - m01 * r1) / det, (m00 * r1 - m01 * r0) / det
        face = torch.stack([1.0 - s - t, s, t], 1)
        best, dist = face, None
        for i, j in ((0, 1), (1, 2), (2, 0)):
            e = X[:, j] - X[:, i]
            q = (((P - X[:, i]) * e).sum(1) / (e * e).sum(1)).clamp(0.0, 1.0)
            b = torch.cat([((1.0 - q) if v == i else q if v == j else 0.0 * q)[:, None] for v in range(3)], 1)
            dd = (P - (b[:, :, None] * X).sum(1)).square().sum(1)
            if dist is None:
                best, dist = b, dd
            else:
                near = dd < dist
                best, dist = torch.where(near[:, None], b, best), torch.where(near, dd, dist)
        inside = (face >= 0.0).all(1)
        return torch.where(inside[:, None], face, best)

    def pairs(self, xg, tri, reach):
        """(flat grid point, triangle) pairs of the triangles' dilated boxes (reach None: all points)."""
        dims = torch.tensor([self.n, self.n, self.nz], device="cuda")
        V = xg[tri.long()]
        if reach is None:
            lo, ext = torch.zeros_like(V[:, 0]).long(), dims.expand(len(tri), 3)
        else:
            lo = torch.ceil((V.amin(1) - reach) / self.dx).long().clamp(min=0)
            ext = (torch.minimum(torch.floor((V.amax(1) + reach) / self.dx).long(), dims - 1) - lo + 1).clamp(min=0)
        cnt = ext.prod(1)
        t = torch.repeat_interleave(torch.arange(len(tri), device="cuda"), cnt)
        l = torch.arange(len(t), device="cuda") - torch.repeat_interleave(cnt.cumsum(0) - cnt, cnt)
        ek, ej = ext[t, 2], ext[t, 1]
        k, j, i = lo[t, 2] + l % ek, lo[t, 1] + (l // ek) % ej, lo[t, 0] + l // (ek * ej)
        return (i * self.n + j) * self.nz + k, t

    def point(self, p):
        return torch.stack([p // (self.n * self.nz), (p // self.nz) % self.n, p % self.nz], 1).double() * self.dx

    def mask_at(self, xw, vw, tri, fr, tanh=False):
        """Band points p with chi and u_s there, differentiable in xw with each
        point's closest triangle held fixed."""
        f8 = dict(device="cuda", dtype=torch.float64)
        R, XO, VO, Om = (torch.as_tensor(np.asarray(fr[k]), **f8) for k in ("R", "X_O", "V_O", "Omega"))
        R = R.reshape(3, 3)
        tw, h = 2.0 * self.dx, 1.5 * self.dx
        xg = XO + xw @ R.T
        with torch.no_grad():
            p, t = self.pairs(xg, tri, None if tanh else tw + h)
            X, P = xg[tri.long()[t]], self.point(p)
            d = (P - (self.closest(P, X)[:, :, None] * X).sum(1)).square().sum(1).sqrt()
            if not tanh:
                near = d < tw + h
                p, t, d = p[near], t[near], d[near]
            u, inv = torch.unique(p, return_inverse=True)
            dmin = torch.full((len(u),), math.inf, **f8).scatter_reduce_(0, inv, d, "amin")
            tie = d <= dmin[inv] * (1.0 + 1e-13)
            win = torch.full((len(u),), len(tri), device="cuda", dtype=torch.long)
            win.scatter_reduce_(0, inv[tie], t[tie], "amin")
        X, P = xg[tri.long()[win]], self.point(u)
        b = self.closest(P, X)
        # a grid point on a node: the weights have no derivative there and the flat profile needs none
        b = torch.where(((P[:, None] - X).square().sum(2) < 1e-24).any(1)[:, None], b.detach(), b)
        d = (P - (b.detach()[:, :, None] * X).sum(1)).square().sum(1).clamp(min=1e-60).sqrt()
        if tanh:
            chi = 0.5 * (1.0 - torch.tanh((d - tw) / h))
        else:
            q = ((d - tw + h) / (2.0 * h)).clamp(0.0, 1.0)
            chi = 0.5 * (1.0 + torch.cos(math.pi * q))
        us = VO + torch.linalg.cross(Om.expand_as(P), P - XO) + ((b[:, :, None] * vw[tri.long()[win]]).sum(1)) @ R.T
        return u, chi, us

    def mask(self, at):
        p, chi, us = at
        n3 = self.n * self.n * self.nz
        f = [torch.zeros(n3, device="cuda", dtype=torch.float64).index_put((p,), v) for v in (chi, us[:, 0], us[:, 1], us[:, 2])]
        shape = (self.n, self.n, self.nz)
        return f[0].view(shape), [f[1].view(shape), f[2].view(shape), f[3].view(shape)]

    def loads(self, pf, xw, tri, fr):
        """Node pressures (smoothed 4-point cosine delta) and node forces -p (A/3) n."""
        f8 = dict(device="cuda", dtype=torch.float64)
        R, XO = torch.as_tensor(np.asarray(fr["R"]), **f8).reshape(3, 3), torch.as_tensor(np.asarray(fr["X_O"]), **f8)
        xg = XO + xw @ R.T
        g = xg / self.dx
        lo = torch.floor(g) - 2
        at = lo[:, :, None] + torch.arange(6, **f8)
        r = (g[:, :, None] - at).abs()
        c, hp = 2.0 / math.pi, 0.5 * math.pi
        w = torch.where(r <= 1.5, 0.25 * (1.0 + c * (torch.sin(hp * (r + 0.5)) - torch.sin(hp * (r - 0.5)))),
                        torch.where(r < 2.5, 0.25 * ((2.5 - r) - c * torch.sin(hp * (r - 0.5))), 0.0 * r))
        i, j, k = at[:, 0].long() % self.n, at[:, 1].long() % self.n, at[:, 2].long() % self.nz
        sub = pf[i[:, :, None, None], j[:, None, :, None], k[:, None, None, :]]
        pn = torch.einsum("vi,vj,vk,vijk->v", w[:, 0], w[:, 1], w[:, 2], sub)
        V = xg[tri.long()]
        area = torch.linalg.cross(V[:, 1] - V[:, 0], V[:, 2] - V[:, 0]) / 6.0
        sums = torch.zeros_like(xg)
        for v in range(3):
            sums.index_add_(0, tri[:, v].long(), area)
        return pn, -pn[:, None] * sums


def exact(case, seed):
    """What ``run`` returns on a fresh state of these inputs, in 64 bits."""
    kind, steps = case["kind"], case["steps"]
    x = _Exact(case)
    if kind == "gradient":
        return _exact_gradient(case, seed, x)
    with torch.no_grad():
        uh = x.velocity_hat(_velocity(case, seed))
        if kind == "fields":
            return torch.stack([x.inv(f) for f in uh])
        if kind == "fsi":
            w = _fsi_wing(case)
            xw, tri = _gpu(w["x0"]), _gpu(w["tri"], torch.int32)
            fr = _frames(0.0)[0]
            chi, us = x.mask(x.mask_at(xw, torch.zeros_like(xw), tri, fr))
            uh, _, _ = x.step(uh, None, chi, us)
            pf = x.pressure(uh, chi, us)
            f = x.loads(pf, xw, tri, fr)[1].cpu().numpy() @ np.asarray(fr["R"], dtype=np.float64).reshape(3, 3)
            return {"p": pf, "f": f, "x": None, "v": None}   # the network's own solution: none in closed form
        if kind in ("decay", "plate"):
            prev, chi, us, fm = None, None, None, None
            if kind == "plate":
                xw, vw, tri, fr = _plate()
                chi, us = x.mask(x.mask_at(_gpu(xw), _gpu(vw), _gpu(tri, torch.int32), fr, tanh=True))
            for _ in range(steps):
                uh, prev, fm = x.step(uh, prev, chi, us)
            u = torch.stack([x.inv(f) for f in uh])
            return u if kind == "decay" else {"force": fm.cpu().numpy(), "u": u}
        tri, xw0, seq = _motion(case, seed, POSITIONS + 1)
        tri = _gpu(tri, torch.int32)
        pos = [(_gpu(q[0]), _gpu(q[1]), tri, q[2]) for q in seq]
        prev, fm = None, []
        if kind == "wing":
            for k in range(steps):
                chi, us = x.mask(x.mask_at(*pos[k % POSITIONS]))
                uh, prev, f = x.step(uh, prev, chi, us)
                fm.append(f)
            del prev, chi, us
            return {"force": torch.stack(fm).cpu().numpy(), "u": torch.stack([x.inv(f) for f in uh])}
        if kind == "pressure":
            chi, us = x.mask(x.mask_at(*pos[0]))
            for _ in range(2):
                uh, prev, _ = x.step(uh, prev, chi, us)
            pf = x.pressure(uh, chi, us)
            pn, fn = x.loads(pf, pos[0][0], tri, pos[0][3])
            return {"p": pf, "p_nodes": pn, "f_nodes": fn}
        # adjoint: one Euler step before the two that are reversed
        chi, us = x.mask(x.mask_at(*pos[0]))
        uh, prev, _ = x.step(uh, None, chi, us)
    w = torch.tensor(ADJ_F + ADJ_M, device="cuda", dtype=torch.float64)
    leaf = [x.mask(x.mask_at(*pos[k + 1])) for k in range(2)]
    for chi, us in leaf:
        for f in [chi] + us:
            f.requires_grad_(True)
    uh2, _, f0 = x.step(uh, prev, *leaf[0])
    f1 = x.force([x.inv(f) for f in uh2], *leaf[1])
    gr = torch.autograd.grad((w * (f0 + f1)).sum(), [f for chi, us in leaf for f in [chi] + us])
    return {"chi": [gr[0], gr[4]], "us": [torch.stack(gr[1:4]), torch.stack(gr[5:8])]}


def _exact_gradient(case, seed, x):
    steps = case["steps"]
    tri, xw0, seq = _motion(case, seed, POSITIONS + 1)
    tri, xw0 = _gpu(tri, torch.int32), _gpu(xw0)
    xw = xw0.clone().requires_grad_(True)
    with torch.no_grad():
        uh = x.velocity_hat(_velocity(case, seed))
    prev, total = None, 0.0
    for k in range(steps):
        q = seq[k % POSITIONS]
        chi, us = x.mask(x.mask_at(xw + (_gpu(q[0]) - xw0), _gpu(q[1]), tri, q[2]))
        uh, prev, f = x.step(uh, prev, chi, us)
        total = total + f
    mean = total / steps
    return {"mean": mean.detach(), "xw": torch.autograd.grad(mean[2], xw)[0]}
