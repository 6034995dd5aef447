"""Pair kernels on tiles 64 sites wide give the bits of the 32 x 8 tiles (a site's arithmetic does not know
its tile): cut tiles, lattices narrower than a tile or its halo, single planes, several z chunks, both
population layouts; and the lattices that take them."""
import numpy as np
import pytest

from tests.helpers import drop_populations, library, make_ctx, oracle_model

pytestmark = pytest.mark.gpu

F32, F16DEV, BF16DEV = 1, 2, 3
D3 = [("D3Q19", "equilibrium", s) for s in [(64, 4, 3), (128, 13, 9), (38, 13, 11), (96, 20, 7), (2, 3, 3), (32, 5, 1),
                                            (130, 10, 40), (66, 9, 33)]]


def _both(lat, scheme, shape, storage, monkeypatch):
    lb = library()
    m = oracle_model(lat, scheme)
    f0 = drop_populations(m, shape, 0.3 * min(shape), perturb=1e-3, seed=41)
    out, forms = [], []
    for wide in ("0", "1"):
        monkeypatch.setenv("LB_WIDE", wide)
        with make_ctx(lb, lat, scheme, shape, storage=storage) as c:
            c.set_populations(f0)
            c.step(5)
            out.append(c.get_populations())
            forms.append(c.kernel_info()["form"])
    assert "32x8" in forms[0] and "64x" in forms[1], forms
    assert np.isfinite(out[0]).all()
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("storage", [F32, F16DEV, BF16DEV])
@pytest.mark.parametrize("lat,scheme,shape", D3)
def test_same_bits(lat, scheme, shape, storage, monkeypatch):
    _both(lat, scheme, shape, storage, monkeypatch)


@pytest.mark.parametrize("lat,scheme,shape,storage,wide", [
    ("D3Q19", "equilibrium", (128, 64, 64), F32, True), ("D3Q19", "equilibrium", (64, 32, 32), F32, False),
    ("D3Q19", "equilibrium", (64, 32, 32), F16DEV, True), ("D3Q19", "equilibrium", (96, 96, 96), F16DEV, False),
    ("D3Q19", "equilibrium", (100, 76, 54), BF16DEV, True)])
def test_which_tile(lat, scheme, shape, storage, wide, monkeypatch):
    monkeypatch.delenv("LB_WIDE", raising=False)
    lb = library()
    with make_ctx(lb, lat, scheme, shape, storage=storage) as c:
        assert ("64x" in c.kernel_info()["form"]) == wide
