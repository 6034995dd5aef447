"""D3Q19 forcing scheme, odd nx: the two-pass form (density field) gives the bits of the one-site fused kernel
that steps such a lattice where no field can be had.  Widths around the tile's 32 sites, lattices narrower
than the halo, single planes and rows, several z chunks."""
import numpy as np
import pytest

from tests.helpers import drop_populations, library, make_ctx, oracle_model

pytestmark = pytest.mark.gpu

F32, F16DEV, BF16DEV = 1, 2, 3


@pytest.mark.parametrize("storage", [F32, F16DEV, BF16DEV])
@pytest.mark.parametrize("shape", [(37, 13, 11), (1, 1, 1), (5, 2, 4), (3, 70, 20), (31, 4, 5), (33, 5, 1), (65, 9, 33),
                                   (101, 75, 53)])
def test_same_bits_as_the_fused_kernel(shape, storage, monkeypatch):
    lb = library()
    m = oracle_model("D3Q19", "forcing")
    f0 = drop_populations(m, shape, 0.3 * min(shape), perturb=1e-3, seed=31)
    out = {}
    for field in ("0", "1"):
        monkeypatch.setenv("LB_D3_FIELD", field)
        with make_ctx(lb, "D3Q19", "forcing", shape, storage=storage) as c:
            c.set_populations(f0)
            c.step(4)
            out[field] = c.get_populations()
            assert ("density field" in c.kernel_info()["form"]) == (field == "1")
    assert np.isfinite(out["0"]).all()
    assert np.array_equal(out["0"], out["1"])
