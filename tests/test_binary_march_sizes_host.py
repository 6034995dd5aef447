"""Which float32 D3Q19 binary lattices run the marching step (fake runtime, by the kernels launched): not the
small ones and, in the equilibrium scheme, not those of fewer than four rows."""
import pytest

from tests import fakecuda

SIZES = [((48, 48, 48), False, False), ((54, 54, 54), False, False), ((60, 60, 60), False, False), ((64, 64, 40), False, False),
         ((65, 50, 50), False, False), ((64, 64, 64), True, True), ((48, 64, 64), True, True), ((101, 75, 53), True, True),
         ((512, 1, 512), True, False), ((512, 3, 200), True, False), ((256, 4, 256), True, True), ((512, 512, 1), True, True)]


@pytest.mark.parametrize("scheme", [0, 1])
def test_sizes(scheme, tmp_path):
    out = fakecuda.run(f"""
got = []
for shape in {[s for s, _, _ in SIZES]}:
    n = fake.fake_launches(b"kernel3_march")
    with lb.BinaryContext(shape, -0.04, 0.04, 0.08, 1.0, 1.0, 1.0, scheme={scheme}, storage=1) as c:
        one = np.ones(c.shape)
        c.init_fields(one, one)
        c.step(1)
    got.append(fake.fake_launches(b"kernel3_march") > n)
print(json.dumps(got))
""", tmp_path)
    assert out == [(f if scheme else e) for _, f, e in SIZES]
