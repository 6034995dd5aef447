"""Contexts near the device's memory limit (fake runtime): the workspace of the step in passes is given back
when a later allocation of the context fails, and the fused kernel steps on."""
import pytest

from tests import fakecuda

# storage, bytes of workspace per site; what the call allocates per site
CALLS = {"fields": ("c.fields()", 96), "populations": ("c.get_populations()", 152), "box": ("c.get_populations_box((0,0,0),(32,32,32))", 152)}


@pytest.mark.parametrize("call", CALLS)
@pytest.mark.parametrize("storage,workspace,passes", [(0, 88, "density3_f64"), (1, 4, "density_pairs"), (2, 4, "density_pairs")])
def test_workspace_is_given_back(storage, workspace, passes, call, tmp_path):
    code, need = CALLS[call]
    out = fakecuda.run(f"""
N = 32 ** 3
c = lb.Context(1, (32, 32, 32), A_VDW, B_VDW, 0.55, 0.01, 0.8, 1, {storage})
c.init_drops([(16, 16, 16)], [8.0])
c.step(70)
form, n = c.kernel_info()["form"], fake.fake_launches(b"{passes}")
fake.fake_capacity(fake.fake_used() + ({need} - 2) * N + 20000)      # {need} bytes per site are not there
st = status(lambda: {code})
info = c.kernel_info()
c.step(70)
print(json.dumps(dict(status=st, before=form, after=info["form"], passes=[n, fake.fake_launches(b"{passes}")],
                      fused=fake.fake_launches(b"step_kernel3d"), ctas=info["ctas"])))
""", tmp_path)
    assert out["status"] == 0, out
    assert "pass" in out["before"] or "density field" in out["before"]
    assert "pass" not in out["after"] and "density field" not in out["after"] and out["ctas"] > 0
    assert out["passes"][0] > 0 and out["passes"][1] == out["passes"][0] and out["fused"] > 0


def test_without_a_workspace_the_call_still_says_so(tmp_path):
    """Nothing to give back: LB_ENOMEM as ever, and the context goes on."""
    out = fakecuda.run("""
c = lb.Context(1, (32, 32, 32), A_VDW, B_VDW, 0.55, 0.01, 0.8, 0, 1)
c.init_drops([(16, 16, 16)], [8.0])
fake.fake_capacity(fake.fake_used() + 1000)
print(json.dumps([status(c.fields), status(c.step, 3), status(c.synchronize)]))
""", tmp_path)
    assert out == [2, 0, 0]


@pytest.mark.parametrize("scheme,storage,nx", [(0, 2, 34), (0, 1, 37), (1, 2, 37), (1, 0, 2)])
def test_a_work_list_beyond_the_hosts_memory_is_an_error_code(scheme, storage, nx, tmp_path):
    """A lattice of hundreds of millions of column tiles under a limit of the process's memory: LB_ENOMEM, no
    exception through the C entry."""
    out = fakecuda.run(f"""
import resource
lb.load_library()
used = int(open("/proc/self/statm").read().split()[0]) * resource.getpagesize()
resource.setrlimit(resource.RLIMIT_AS, (used + 400_000_000,) * 2)
st = status(lb.Context, 1, ({nx}, {2_000_000_000 // nx}, 1), A_VDW, B_VDW, 0.55, 0.01, 0.8, {scheme}, {storage}, buffer=(1 << 20, 1 << 50))
one = status(lb.work_list, 152, 2, ({nx}, {2_000_000_000 // nx}, 1), (1, 1))
print(json.dumps([st, one]))
""", tmp_path)
    assert out == [2, 2]
