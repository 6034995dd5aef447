"""The marching float32 D3Q19 binary step beside the brick kernel it replaces on larger lattices, on
cut tiles, odd widths, lattices narrower than the halo, single planes and several z chunks: after
20 steps its error against the float64 oracle (2-norm, relative) is at most one and a half times
the brick kernel's, or eight float32 roundings."""
import numpy as np
import pytest

from oracle import binary_oracle as BO
from tests.helpers import library

pytestmark = pytest.mark.gpu


def _off(got, want):
    return np.linalg.norm(got - want) / np.linalg.norm(want)


@pytest.mark.parametrize("scheme", ["equilibrium", "forcing"])
@pytest.mark.parametrize("shape", [(34, 10, 9), (33, 9, 8), (64, 8, 40), (2, 3, 3), (1, 1, 1), (5, 2, 4), (38, 21, 1)])
def test_against_brick_kernel(shape, scheme, monkeypatch):
    lb = library()
    m = BO.BinaryModel("D3Q19", -0.04, 0.04, 0.08, 0.7, 0.8, 0.9, scheme=scheme)
    nx, ny, nz = shape
    rng = np.random.default_rng(13)
    rho0 = 1 + 1e-2 * rng.uniform(-1, 1, (nz, ny, nx))
    phi0 = BO.drop_phi((nz, ny, nx), [(nx / 2, ny / 2, nz / 2)], [0.3 * max(shape)], 1.0, -1.0, 2.0)
    u0 = [1e-2 * rng.uniform(-1, 1, rho0.shape) for _ in range(3)]
    f, g = BO.init_equilibrium(rho0, phi0, m, u0)
    want = BO.run(f, g, m, 20)
    off = {}
    for march in ("1", "0"):
        monkeypatch.setenv("LB_B3_MARCH", march)
        with lb.BinaryContext(shape, m.A, m.B, m.kappa, m.Gamma, m.tau, m.tau_phi,
                              scheme=lb.FORCING if scheme == "forcing" else lb.EQUILIBRIUM, storage=lb.F32) as c:
            c.set_populations(f, g)
            c.step(20)
            off[march] = [_off(got, w) for got, w in zip(c.get_populations(), want)]
    for march, brick in zip(off["1"], off["0"]):
        assert march <= max(1.5 * brick, 8 * 2.0 ** -24)
