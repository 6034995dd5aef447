"""The float64 D2Q9 step takes its tile by the lattice's size (8 x 4, 8 x 8 or 32 x 8 sites): one
step of a perturbed drop against the oracle at sizes on both sides of each line, with ragged
tiles, to the float64 parity bound."""
import numpy as np
import pytest

from oracle import lb_oracle as O
from tests.helpers import drop_populations, library, make_ctx, oracle_model, rel_inf

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scheme", ["equilibrium", "forcing"])
@pytest.mark.parametrize("shape", [(8, 4), (9, 5), (1, 7), (181, 180), (183, 179), (445, 444), (447, 443), (33, 6001),
                                   (6001, 34)])
def test_one_step(shape, scheme):
    lb = library()
    m = oracle_model("D2Q9", scheme)
    f0 = drop_populations(m, shape, 0.3 * min(shape), perturb=1e-3, seed=21)
    with make_ctx(lb, "D2Q9", scheme, shape) as c:
        c.set_populations(f0)
        c.step(1)
        got = c.get_populations()
        tile = tuple(c.kernel_info()["tile"])
    assert rel_inf(got, O.step(f0, m)) < 1e-12
    sites = shape[0] * shape[1]
    if sites < 30000:
        assert tile == (8, 4)
    if sites > 210000:
        assert tile == (32, 8)
