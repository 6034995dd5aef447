"""Rounding of the float64 D3Q19 step in passes: after one step its populations are no further from the
oracle's formulas in extended precision (2-norm over all populations) than the fused kernel's, which divides
once for each reciprocal."""
import dataclasses
from fractions import Fraction

import numpy as np
import pytest

from oracle import lb_oracle as O
from tests.helpers import drop_populations, library, make_ctx, oracle_model

pytestmark = pytest.mark.gpu

LD = np.longdouble


def _extended(o):
    """The model's coefficients (fractions with small denominators) and parameters in extended precision."""
    for fld in dataclasses.fields(o):
        v = getattr(o, fld.name)
        if dataclasses.is_dataclass(v):
            _extended(v)
        elif isinstance(v, float):
            fr = Fraction(v).limit_denominator(10000)
            coefficient = fld.name not in ("a", "b", "T", "kappa", "tau")
            setattr(o, fld.name, LD(fr.numerator) / LD(fr.denominator) if coefficient else LD(v))
        elif isinstance(v, np.ndarray) and v.dtype == np.float64:
            fr = [Fraction(float(x)).limit_denominator(10000) for x in v.ravel()]
            setattr(o, fld.name, np.array([LD(f.numerator) / LD(f.denominator) for f in fr], dtype=LD).reshape(v.shape))
    return o


@pytest.mark.skipif(np.finfo(LD).eps > 1e-18, reason="no extended precision on this machine")
@pytest.mark.parametrize("scheme", ["forcing", "equilibrium"])
@pytest.mark.parametrize("T,kappa,tau", [(0.55, 0.01, 0.8), (0.56, 0.025, 1.0), (0.53, 0.005, 1.2), (0.55, 0.015, 0.7)])
def test_no_further_off_than_the_fused_kernel(scheme, T, kappa, tau, monkeypatch):
    lb = library()
    shape = (20, 18, 16)
    m = oracle_model("D3Q19", scheme, T=T, kappa=kappa, tau=tau)
    f0 = drop_populations(m, shape, 5.0, perturb=1e-3, seed=7)
    want = O.run(f0.astype(LD), _extended(m), 1)
    assert want.dtype == LD
    off = {}
    for slab in (None, "0"):
        if slab is not None:
            monkeypatch.setenv("LB_F64_SLAB", slab)
        with make_ctx(lb, "D3Q19", scheme, shape, T=T, kappa=kappa, tau=tau) as c:
            c.set_populations(f0)
            c.step(1)
            off[slab] = float(np.sqrt(((c.get_populations().astype(LD) - want) ** 2).sum()))
            assert ("passes" in c.kernel_info()["form"]) == (slab is None)
    assert off[None] <= off["0"], off
