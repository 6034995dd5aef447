"""Rounding of the marching float32 D3Q19 binary step: against the float64 oracle (2-norm of f and of g) it is
no further off than the brick kernel, after one step and after twenty, for relaxation times of one (where a
population is its equilibrium) and others."""
import numpy as np
import pytest

from oracle import binary_oracle as BO
from tests.helpers import library

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scheme", ["equilibrium", "forcing"])
@pytest.mark.parametrize("Gamma,tau,tau_phi", [(1.0, 1.0, 1.0), (0.7, 0.8, 0.9), (1.3, 1.2, 0.8)])
@pytest.mark.parametrize("shape", [(40, 36, 33), (33, 20, 27)])
def test_no_further_off_than_the_bricks(shape, Gamma, tau, tau_phi, scheme, monkeypatch):
    lb = library()
    m = BO.BinaryModel("D3Q19", -0.04, 0.04, 0.08, Gamma, tau, tau_phi, scheme=scheme)
    nx, ny, nz = shape
    rng = np.random.default_rng(5)
    rho0 = 1 + 1e-3 * rng.uniform(-1, 1, (nz, ny, nx))
    phi0 = BO.drop_phi((nz, ny, nx), [(nx / 2, ny / 2, nz / 2)], [0.3 * min(shape)], 1.0, -1.0, 2.0)
    f, g = BO.init_equilibrium(rho0, phi0, m, [np.zeros_like(rho0)] * 3)
    want = {1: BO.run(f, g, m, 1)}
    want[20] = BO.run(*want[1], m, 19)
    off = {}
    for march in ("1", "0"):
        monkeypatch.setenv("LB_B3_MARCH", march)
        with lb.BinaryContext(shape, m.A, m.B, m.kappa, m.Gamma, m.tau, m.tau_phi,
                              scheme=lb.FORCING if scheme == "forcing" else lb.EQUILIBRIUM, storage=lb.F32) as c:
            c.set_populations(f, g)
            done, off[march] = 0, []
            for steps in (1, 20):
                c.step(steps - done)
                done = steps
                off[march] += [np.linalg.norm(got - w) for got, w in zip(c.get_populations(), want[steps])]
    assert all(a <= b for a, b in zip(off["1"], off["0"])), off
