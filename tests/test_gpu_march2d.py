"""The marching form of the D2Q9 equilibrium step in 16-bit storage gives the bits of the tiles: strips
cut by the lattice's edge, lattices narrower than a strip or its halo, chunks of one row, of all
rows and with a ragged end; and the chunk that larger lattices take."""
import numpy as np
import pytest

from tests.helpers import drop_populations, library, make_ctx, oracle_model

pytestmark = pytest.mark.gpu

F16DEV, BF16DEV = 2, 3


@pytest.mark.parametrize("storage", [F16DEV, BF16DEV])
@pytest.mark.parametrize("shape", [(60, 12), (62, 13), (2, 5), (4, 1), (46, 37), (178, 9), (256, 40)])
def test_same_bits_as_tiles(shape, storage, monkeypatch):
    lb = library()
    m = oracle_model("D2Q9", "equilibrium")
    f0 = drop_populations(m, shape, 0.3 * min(shape), perturb=1e-3, seed=17)
    out = {}
    for rows in (0, 1, 3, 8, shape[1]):
        monkeypatch.setenv("LB_D2_ROWS", str(rows))
        with make_ctx(lb, "D2Q9", "equilibrium", shape, storage=storage) as c:
            c.set_populations(f0)
            c.step(5)
            out[rows] = c.get_populations()
            assert ("marching" in c.kernel_info()["form"]) == (rows > 0)
    for rows, got in out.items():
        assert np.array_equal(got, out[0]), rows


@pytest.mark.parametrize("shape,march", [((2048, 2048), True), ((4096, 500), True), ((1100, 1100), True), ((1024, 1024), False),
                                         ((2047, 2048), False)])
def test_which_form(shape, march, monkeypatch):
    monkeypatch.delenv("LB_D2_ROWS", raising=False)
    lb = library()
    out = {}
    for rows in (None, "0"):
        if rows is not None:
            monkeypatch.setenv("LB_D2_ROWS", rows)
        with make_ctx(lb, "D2Q9", "equilibrium", shape, storage=F16DEV) as c:
            c.init_drops([(shape[0] / 2, shape[1] / 2)], [0.2 * min(shape)])
            c.step(2)
            out[rows] = c.get_state()
            assert ("marching" in c.kernel_info()["form"]) == (march and rows is None)
    assert out[None] == out["0"]
