"""Contexts where no CUDA device can be used (fake runtime): an error code for every lattice, scheme and
storage, no crash on the way to it."""
from tests import fakecuda


def test_create_returns_an_error_code(tmp_path):
    out = fakecuda.run("""
fake.fake_no_device(1)
got = {}
for lat, shape in ((0, (512, 512)), (0, (64, 20000)), (0, (37, 11)), (1, (64, 32, 32)), (1, (37, 9, 8))):
    for scheme in (0, 1):
        for storage in (0, 1, 2, 3):
            got[f"{lat} {shape} {scheme} {storage}"] = status(lb.Context, lat, shape, A_VDW, B_VDW, 0.55, 0.01, 0.8, scheme, storage)
for shape, storage in (((64, 64), 2), ((64, 64, 64), 1), ((64, 64, 64), 0)):
    got[f"binary {shape} {storage}"] = status(lb.BinaryContext, shape, -0.04, 0.04, 0.08, 1.0, 1.0, 1.0, storage=storage)
print(json.dumps(got))
""", tmp_path)
    assert len(out) == 43
    # LB_ENOMEM: the population buffers cannot be had; a binary context says LB_ECUDA
    assert out == {k: 3 if k.startswith("binary") else 2 for k in out}
