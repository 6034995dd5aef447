"""Which D3Q19 equilibrium lattices run tiles of 64 x 4 sites (fake runtime: 152 SMs): not those that such
tiles were measured to slow down."""
from tests import fakecuda

F32, F16DEV, BF16DEV = 1, 2, 3
WIDE = [((128, 128, 128), F16DEV, True), ((100, 76, 54), BF16DEV, True), ((224, 224, 224), F16DEV, True),
        ((288, 232, 50), F16DEV, True), ((288, 200, 100), F16DEV, False), ((160, 160, 160), F16DEV, False),
        ((144, 144, 144), F16DEV, False), ((138, 158, 13), F16DEV, False), ((96, 96, 96), F16DEV, False),
        ((32, 4, 4096), F16DEV, False), ((160, 160, 160), BF16DEV, False), ((34, 51, 207), F16DEV, True),
        ((146, 36, 26), F16DEV, False), ((288, 263, 12), F16DEV, False), ((200, 5, 84), F16DEV, False),
        ((510, 6, 177), F16DEV, False), ((510, 6, 177), F32, False), ((296, 6, 162), F32, False), ((512, 4, 256), F16DEV, True),
        ((288, 288, 288), F16DEV, True), ((512, 512, 512), F16DEV, True), ((96, 4, 2048), F32, True),
        ((128, 128, 128), F32, True), ((144, 144, 144), F32, True), ((288, 288, 288), F32, True), ((146, 246, 39), F32, True),
        ((48, 48, 48), F32, False), ((160, 160, 160), F32, False), ((138, 158, 13), F32, False), ((160, 25, 68), F32, False),
        ((138, 97, 48), F32, False), ((338, 13, 58), F32, False), ((160, 293, 12), F32, True), ((512, 512, 512), F32, True),
        ((97, 100, 100), F32, False)]


def test_which_tile(tmp_path):
    out = fakecuda.run(f"""
got = []
for shape, storage, _ in {WIDE!r}:
    with lb.Context(1, shape, A_VDW, B_VDW, 0.55, 0.01, 0.8, 0, storage, buffer=(1 << 20, 1 << 50)) as c:
        got.append("64x4" in c.kernel_info()["form"])
print(json.dumps(got))
""", tmp_path)
    assert out == [w for _, _, w in WIDE], [s for s, w in zip(WIDE, out) if s[2] != w]
