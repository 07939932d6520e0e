"""Force and moment of the last step do not depend on what is read between the
step and ps_forces: diagnostics, velocity, mask, pressure and a saved state
leave them bit for bit."""
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
@pytest.mark.parametrize("n,nz", [(12, 12), (32, 16), (48, 48)])
def test_forces_survive_other_reads(n, nz, prec):
    L = 4.0
    dt = torch.float64 if prec == "fp64" else torch.float32
    d = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to("cuda", dt)  # noqa: E731
    g = Solver(n, L, 0.01, 0.1, 1e-3, precision=prec, nz=nz)
    g.set_velocity(d(inputs.random_field(n, L, seed=8, rms=0.3, nz=nz)))
    rng = np.random.default_rng(n)
    chi = np.zeros((n, n, nz))
    chi[n // 4: n // 2, n // 3: n // 2 + 1, 1: nz // 2] = 0.7
    g.set_mask(d(chi), d(0.1 * rng.standard_normal((3, n, n, nz))))
    g.step(1)
    want = np.concatenate(g.forces())
    assert np.all(np.isfinite(want)) and np.all(want != 0.0)
    for read in (g.diagnostics, g.velocity, g.mask, g.pressure, lambda: g.save_state(g.state_buffer())):
        read()
        assert np.array_equal(np.concatenate(g.forces()), want)
    g.close()
