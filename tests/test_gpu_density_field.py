"""The D3Q19 forcing step in two passes (density field, then collision) against the fused kernels:
the same bits as the fused pair kernel (even nx), the oracle's step where the fused form is the
one-site kernel (odd nx).  Lattices narrower than the halo, cut tiles, single planes, several z
chunks, both population layouts; and the lines between the two forms."""
import numpy as np
import pytest

from oracle import lb_oracle as O
from tests.helpers import drop_populations, library, make_ctx, oracle_model, rel_inf

pytestmark = pytest.mark.gpu

F32, F16DEV, BF16DEV = 1, 2, 3
SHAPES = [(38, 13, 11), (64, 16, 9), (96, 20, 7), (2, 3, 3), (32, 5, 1), (130, 10, 40), (37, 13, 11), (1, 1, 1), (5, 2, 4),
          (65, 9, 33)]


@pytest.mark.parametrize("storage,tol", [(F32, 2e-6), (F16DEV, 1e-5), (BF16DEV, 8e-5)])
@pytest.mark.parametrize("shape", SHAPES)
def test_both_forms(shape, storage, tol, monkeypatch):
    lb = library()
    m = oracle_model("D3Q19", "forcing")
    f0 = drop_populations(m, shape, 0.3 * min(shape), perturb=1e-3, seed=31)
    out, steps = {}, 4
    for field in ("1", "0"):
        monkeypatch.setenv("LB_D3_FIELD", field)
        with make_ctx(lb, "D3Q19", "forcing", shape, storage=storage) as c:
            c.set_populations(f0)
            start = c.get_populations()
            c.step(steps)
            out[field] = c.get_populations()
            assert ("density field" in c.kernel_info()["form"]) == (field == "1")
    if shape[0] % 2 == 0:
        assert np.array_equal(out["1"], out["0"])
    else:       # per step the bound of the pair kernels' parity tests
        assert rel_inf(out["1"], O.run(start, m, steps)) < steps * tol


@pytest.mark.parametrize("shape,storage,field", [((24, 24, 24), F32, True), ((360, 360, 320), F32, False),
                                                 ((96, 96, 96), F16DEV, True), ((160, 160, 160), F16DEV, False),
                                                 ((100, 20, 10), BF16DEV, True), ((101, 20, 10), F32, True)])
def test_which_form(shape, storage, field, monkeypatch):
    monkeypatch.delenv("LB_D3_FIELD", raising=False)
    lb = library()
    with make_ctx(lb, "D3Q19", "forcing", shape, storage=storage) as c:
        assert ("density field" in c.kernel_info()["form"]) == field
