"""Which lattices the marching D2Q9 form takes (fake runtime: 152 SMs): not widths whose last strip of 60 columns
overhangs the lattice much further than a tile of 32 columns would, and not flat ones whose chunks of rows
leave an SM one warp too many."""
from tests import fakecuda

MARCH = {16: False, 30: False, 32: False, 34: True, 48: True, 60: True, 62: False, 64: False, 96: False, 110: True, 120: True,
         124: False, 128: False, 160: True, 180: True, 192: False, 240: True, 256: True, 512: True, 2048: True, 63: False, 2047: False}


def test_widths(tmp_path):
    out = fakecuda.run(f"""
got = {{}}
for nx in {sorted(MARCH)}:
    with lb.Context(0, (nx, 4_200_000 // nx), A_VDW, B_VDW, 0.55, 0.01, 0.8, 0, lb.F16DEV) as c:
        got[nx] = "marching" in c.kernel_info()["form"]
print(json.dumps(got))
""", tmp_path)
    assert {int(k): v for k, v in out.items()} == MARCH


FLAT = [((100000, 12), True), ((80000, 15), False), ((60000, 20), True), ((40000, 30), False), ((20000, 64), True),
        ((3000, 400), True), ((1100, 1100), True), ((1024, 1024), False), ((2048, 2048), True),
        ((2, 600000), True), ((64, 600000), True), ((64, 500000), False)]      # tiles have no launch for 600000 rows


def test_flat_and_tall(tmp_path):
    out = fakecuda.run(f"""
got = []
for shape in {[s for s, _ in FLAT]}:
    with lb.Context(0, shape, A_VDW, B_VDW, 0.55, 0.01, 0.8, 0, lb.BF16DEV, buffer=(1 << 20, 1 << 50)) as c:
        got.append("marching" in c.kernel_info()["form"])
print(json.dumps(got))
""", tmp_path)
    assert out == [m for _, m in FLAT], list(zip(FLAT, out))
