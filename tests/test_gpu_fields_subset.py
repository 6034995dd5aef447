"""lb_fields, lb_batch_fields and lb_binary_fields compute only the outputs that are asked for:
every subset gives the same bits as the full call, and the density sums are exact conversions
(subnormal and zero populations among them)."""
import ctypes as C

import numpy as np
import pytest

from tests.helpers import A_VDW, B_VDW, library, make_ctx

pytestmark = pytest.mark.gpu


def _ptr(a):
    return None if a is None else a.ctypes.data_as(C.POINTER(C.c_double))


@pytest.mark.parametrize("lat,shape", [("D2Q9", (45, 33)), ("D3Q19", (32, 9, 7))])
@pytest.mark.parametrize("scheme", ["equilibrium", "forcing"])
@pytest.mark.parametrize("storage", ["f64", "f32", "f16dev", "bf16dev"])
def test_single_lattice(lat, shape, scheme, storage):
    lb = library()
    with make_ctx(lb, lat, scheme, shape, storage=lb.STORAGE_NAMES[storage]) as c:
        c.init_drops([tuple(n / 2 for n in shape)], [0.3 * min(shape)])
        c.step(3)
        rho, u, v = c.fields()
        for want in ((1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 0, 1)):
            out = [np.empty_like(a) if w else None for a, w in zip((rho, u, v), want)]
            lb._check(c._lib.lb_fields(c._h, *(_ptr(a) for a in out)))
            for a, b in zip(out, (rho, u, v)):
                assert a is None or np.array_equal(a, b)


@pytest.mark.parametrize("storage", ["f64", "f32", "f16dev"])
def test_batch_density_alone(storage):
    lb = library()
    inst = [dict(nx=n, ny=n - 3, T=0.55, kappa=0.01, tau=0.9, radius=0.3 * n) for n in (64, 71)]
    with lb.Batch(inst, A_VDW, B_VDW, lb.FORCING, lb.STORAGE_NAMES[storage]) as b:
        b.init_drops()
        for steps in (0, 3):
            b.step(steps)
            for k in range(2):
                rho, u = b.fields(k)
                alone = np.empty_like(rho)
                lb._check(b._lib.lb_batch_fields(b._h, k, _ptr(alone), None))
                assert np.array_equal(alone, rho)
        # a retired instance is read from the buffer it stopped in
        b.run_to_steady(tol=1e30, every=2, max_steps=4)
        b.step(1)
        rho, u = b.fields(0)
        assert np.isfinite(rho).all() and abs(rho.sum() / b.populations(0).sum() - 1) < 1e-12


@pytest.mark.parametrize("shape,storage", [((46, 21), "f64"), ((46, 21), "f32"), ((45, 21), "f32"), ((46, 21), "f16dev"),
                                           ((33, 9, 6), "f64"), ((33, 9, 6), "f32")])
@pytest.mark.parametrize("scheme", ["equilibrium", "forcing"])
def test_binary(shape, storage, scheme):
    lb = library()
    rng = np.random.default_rng(5)
    with lb.BinaryContext(shape, -0.04, 0.04, 0.08, 0.7, 0.8, 0.9, scheme=lb.FORCING if scheme == "forcing" else
                          lb.EQUILIBRIUM, storage=lb.STORAGE_NAMES[storage]) as c:
        c.init_fields(1 + 0.01 * rng.random(c.shape), rng.uniform(-1, 1, c.shape))
        c.step(2)
        full = c.fields()
        for want in ((1, 1, 0, 0, 0), (0, 0, 1, 0, 0), (0, 0, 0, 1, 0), (0, 0, 0, 0, 1), (1, 0, 0, 1, 0)):
            out = [np.empty_like(a) if w else None for a, w in zip(full, want)]
            lb._check(c._lib.lb_binary_fields(c._h, *(_ptr(a) for a in out)))
            for a, b in zip(out, full):
                assert a is None or np.array_equal(a, b)


@pytest.mark.parametrize("shape", [(40, 12), (33, 8, 5)])
def test_density_sum_of_small_values(shape):
    lb = library()
    rng = np.random.default_rng(7)
    with lb.BinaryContext(shape, -0.04, 0.04, 0.08, 0.7, 0.8, 0.9, storage=lb.F32) as c:
        f = rng.uniform(0.01, 0.1, (c.q,) + c.shape).astype(np.float32)
        g = (rng.uniform(-1, 1, f.shape) * 10.0 ** rng.integers(-45, 3, f.shape)).astype(np.float32)
        g[:, ..., 0] = 0.0
        c.set_populations(f, g)
        rho, phi = c.fields()[:2]
    for got, p in ((rho, f), (phi, g)):
        want = np.zeros(c.shape)
        for i in range(c.q):
            want = want + p[i].astype(np.float64)     # the kernels' order: exact conversions, one rounding per addition
        assert np.array_equal(got, want)
