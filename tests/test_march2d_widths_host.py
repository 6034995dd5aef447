"""Which widths the marching D2Q9 form takes (fake runtime: 152 SMs): not those whose last strip of 60 columns
overhangs the lattice much further than a tile of 32 columns would."""
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
