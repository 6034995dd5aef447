"""Which D3Q19 forcing lattices step over a density field (fake runtime): not those that were measured to be
faster in the fused kernel, and every odd width."""
from tests import fakecuda

F32, F16DEV, BF16DEV = 1, 2, 3
FIELD = [((128, 128, 128), F32, True), ((256, 256, 256), F32, True), ((336, 336, 336), F32, True), ((384, 384, 384), F32, False),
         ((210, 210, 210), F32, True), ((250, 250, 250), F32, False), ((300, 300, 300), F32, False), ((310, 310, 310), F32, False),
         ((32, 120, 120), F32, True), ((32, 200, 200), F32, False), ((24, 300, 300), F32, False), ((16, 400, 400), F32, True),
         ((64, 120, 120), F32, True), ((64, 200, 200), F32, False), ((62, 330, 330), F32, False), ((56, 330, 330), F32, True),
         ((96, 300, 300), F32, True), ((34, 430, 430), F32, True),
         ((128, 128, 128), F16DEV, True), ((512, 512, 512), F16DEV, False), ((300, 300, 300), F16DEV, True),
         ((500, 500, 500), BF16DEV, True), ((32, 120, 120), F16DEV, True), ((32, 300, 300), F16DEV, False),
         ((64, 200, 200), F16DEV, False), ((52, 330, 330), BF16DEV, False), ((30, 300, 300), F16DEV, False),
         ((34, 430, 430), F16DEV, True), ((24, 430, 430), F16DEV, True), ((100, 330, 330), F16DEV, True),
         ((101, 75, 53), BF16DEV, True), ((481, 480, 480), F16DEV, True), ((31, 300, 300), F32, True), ((301, 301, 301), F32, True)]


def test_which_form(tmp_path):
    out = fakecuda.run(f"""
got = []
for shape, storage, _ in {FIELD!r}:
    with lb.Context(1, shape, A_VDW, B_VDW, 0.55, 0.01, 0.8, 1, storage, buffer=(1 << 20, 1 << 50)) as c:
        got.append("density field" in c.kernel_info()["form"])
print(json.dumps(got))
""", tmp_path)
    assert out == [f for _, _, f in FIELD], [c for c, f in zip(FIELD, out) if c[2] != f]
