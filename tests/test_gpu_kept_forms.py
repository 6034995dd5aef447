"""The fused D3Q19 forcing kernels that small lattices no longer run by themselves, against the oracle: the pair
kernel (even nx, both population layouts) and the one-site kernel (odd nx), which step a lattice whose density
field cannot be had, and the pair kernel the large lattices."""
import pytest

from oracle import lb_oracle as O
from tests.helpers import drop_populations, library, make_ctx, oracle_model, rel_inf

pytestmark = pytest.mark.gpu

F32, F16DEV, BF16DEV = 1, 2, 3


# one step from the context's own rounded state: the bounds of test_gpu_parity.test_pair_kernel_parity
@pytest.mark.parametrize("storage,tol", [(F32, 2e-6), (F16DEV, 1e-5), (BF16DEV, 8e-5)])
@pytest.mark.parametrize("shape", [(68, 20, 12), (64, 16, 9), (96, 20, 7), (38, 13, 11), (2, 3, 3), (37, 13, 11), (65, 9, 33),
                                   (5, 2, 4)])
def test_fused_forcing_against_the_oracle(shape, storage, tol, monkeypatch):
    monkeypatch.setenv("LB_D3_FIELD", "0")
    lb = library()
    m = oracle_model("D3Q19", "forcing")
    with make_ctx(lb, "D3Q19", "forcing", shape, storage=storage) as c:
        assert "field" not in c.kernel_info()["form"]
        c.set_populations(drop_populations(m, shape, 0.3 * min(shape), perturb=1e-3, seed=12))
        start = c.get_populations()
        for steps in (1, 4):
            c.step(steps - (0 if steps == 1 else 1))
            assert rel_inf(c.get_populations(), O.run(start, m, steps)) < steps * tol
