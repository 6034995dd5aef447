"""The float64 D3Q19 step in passes: its workspace holds the whole lattice or slabs of planes with
halo planes.  Slabs of any depth give the bits of the whole lattice, and both agree with the fused
kernel (taken where the workspace cannot be had) and with the oracle to the float64 bound."""
import numpy as np
import pytest

from oracle import lb_oracle as O
from tests.helpers import drop_populations, library, make_ctx, oracle_model, rel_inf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scheme", ["equilibrium", "forcing"])
@pytest.mark.parametrize("shape", [(37, 13, 11), (32, 8, 3), (2, 3, 4), (5, 1, 2), (1, 1, 1), (9, 6, 21)])
def test_slabs(shape, scheme, monkeypatch):
    lb = library()
    m = oracle_model("D3Q19", scheme)
    f0 = drop_populations(m, shape, 0.3 * max(shape), perturb=1e-3, seed=8)
    out = {}
    for slab in (None, 1, 2, 3, shape[2] - 1, shape[2], 0):
        if slab is None:
            monkeypatch.delenv("LB_F64_SLAB", raising=False)
        else:
            monkeypatch.setenv("LB_F64_SLAB", str(slab))
        with make_ctx(lb, "D3Q19", scheme, shape) as c:
            c.set_populations(f0)
            c.step(3)
            out[slab] = c.get_populations()
            form = c.kernel_info()["form"]
        assert ("passes" in form) == (slab != 0)
    want = O.run(f0, m, 3)
    for slab, got in out.items():
        assert rel_inf(got, want) < 3e-12, slab
        if slab != 0:
            assert np.array_equal(got, out[None]), slab
