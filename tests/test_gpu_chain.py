"""Chained launches: a step's kernel starts as its predecessor's last CTA leaves, and must still see all
of that kernel's writes.  Runs of steps without a pause give the bits of runs that wait after every
step, on lattices of one CTA, of part of a wave and of several waves; and steps captured in a graph of
the caller between a copy and a kernel give those of plain calls."""
import numpy as np
import pytest
import torch

from tests.helpers import library, make_ctx

pytestmark = pytest.mark.gpu

STEPS = 60   # fewer than a replayed graph holds
CASES = [("D2Q9", (20, 12)), ("D2Q9", (100, 100)), ("D2Q9", (300, 301)), ("D2Q9", (1300, 1200)),
         ("D3Q19", (12, 10, 8)), ("D3Q19", (33, 30, 20)), ("D3Q19", (64, 64, 64))]


@pytest.mark.parametrize("scheme", ["equilibrium", "forcing"])
@pytest.mark.parametrize("storage", [0, 1, 2])
@pytest.mark.parametrize("lat,shape", CASES)
def test_steps_without_a_pause(lat, shape, storage, scheme):
    lb = library()
    out = []
    for pause in (True, False):
        with make_ctx(lb, lat, scheme, shape, storage=storage) as c:
            c.init_drops([[s / 2 for s in shape]], [0.3 * min(shape)])
            for _ in range(STEPS):
                c.step(1)
                if pause:
                    c.synchronize()
            out.append(c.get_populations())
    assert np.isfinite(out[0]).all()
    assert np.array_equal(out[0], out[1])


@pytest.mark.parametrize("scheme", [0, 1])
@pytest.mark.parametrize("shape,storage", [((50, 33), 0), ((200, 100), 1), ((64, 50), 2), ((20, 12, 9), 0),
                                           ((30, 21, 18), 1), ((64, 64, 64), 1)])
def test_binary_steps_without_a_pause(shape, storage, scheme):
    lb = library()
    phi = np.random.default_rng(5).uniform(-1, 1, shape[::-1])
    out = []
    for pause in (True, False):
        with lb.BinaryContext(shape, -0.04, 0.04, 0.08, 0.7, 0.8, 0.9, scheme=scheme, storage=storage) as c:
            c.init_fields(np.ones(shape[::-1]), phi)
            for _ in range(STEPS):
                c.step(1)
                if pause:
                    c.synchronize()
            out.append(c.get_populations())
    for a, b in zip(*out):
        assert np.isfinite(a).all()
        assert np.array_equal(a, b)


@pytest.mark.parametrize("lat,shape,storage", [("D2Q9", (100, 100), 0), ("D2Q9", (128, 64), 1),
                                               ("D3Q19", (33, 30, 20), 1), ("D3Q19", (24, 20, 16), 0)])
def test_steps_in_the_callers_graph(lat, shape, storage):
    lb = library()
    out = []
    for captured in (False, True):
        st = torch.cuda.Stream()
        with make_ctx(lb, lat, "forcing", shape, storage=storage, stream=st.cuda_stream) as c:
            c.init_drops([[s / 2 for s in shape]], [0.3 * min(shape)])
            c.step(2)
            c.synchronize()
            x = torch.zeros(1 << 20, device="cuda")
            y = torch.ones(1 << 20, device="cuda")
            torch.cuda.synchronize()
            if captured:
                g = torch.cuda.CUDAGraph()
                with torch.cuda.graph(g, stream=st):
                    x.copy_(y)
                    c.step(10)
                    x.add_(1.0)
                with torch.cuda.stream(st):
                    for _ in range(3):
                        g.replay()
            else:
                c.step(30)
            c.synchronize()
            out.append(c.get_populations())
    assert np.isfinite(out[0]).all()
    assert np.array_equal(out[0], out[1])
