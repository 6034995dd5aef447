"""lb_ws_train when a CUDA call fails (fake runtime, no GPU): the parameters stay as they were."""
import pytest

from tests import fakecuda

TRAIN = """
n, H, W = 4, 16, 16
ws = lb.WarmStart(seed=1)
before = ws.get_params()
x, t = np.zeros((n, 5, H, W), np.float32), np.zeros((n, 3, H, W), np.float32)
"""


def test_no_optimiser_step_without_gradients(tmp_path):
    """The workspace of the gradients' partial sums cannot be had: LB_ENOMEM, and no optimiser step on the
    gradient buffer that nothing has written."""
    out = fakecuda.run(TRAIN + """
fake.fake_capacity(fake.fake_used() + 12_000_000)      # enough for everything but the partial sums (26 MB)
s = status(ws.train, x, t, epochs=2, batch=2, lr=1e-3)
print(json.dumps(dict(status=s, adam=fake.fake_launches(b"adam"), forward=fake.fake_launches(b"conv_tile"))))
""", tmp_path)
    assert out == dict(status=2, adam=0, forward=0)


@pytest.mark.parametrize("kernel,after,adam", [("gather_batch", 0, 0), ("conv_tile", 2, 0), ("conv_bwd_weight", 1, 0),
                                               ("reduce_grads", 0, 0), ("gather_batch", 1, 1), ("adam_pack", 3, 3)])
def test_a_refused_launch_ends_the_training(kernel, after, adam, tmp_path):
    """A launch that the runtime refuses (in the first minibatch, a later one, the last Adam step): LB_ECUDA, no
    optimiser step after it, and no error left behind for the next call."""
    out = fakecuda.run(TRAIN + f"""
fake.fake_fail_kernel(b"{kernel}", {after})
s = status(ws.train, x, t, epochs=2, batch=2, lr=1e-3)
fake.fake_fail_kernel(b"", 0)
n_adam = fake.fake_launches(b"adam")
again = status(ws.train, x, t, epochs=1, batch=2, lr=1e-3)
print(json.dumps(dict(status=s, adam=n_adam, again=again)))
""", tmp_path)
    assert out == dict(status=3, adam=adam, again=0)


def test_a_refused_launch_fails_the_gradient_call(tmp_path):
    out = fakecuda.run(TRAIN + """
fake.fake_fail_kernel(b"conv_tile", 1)
s = status(ws.loss_grad, x, t)
fake.fake_fail_kernel(b"", 0)
print(json.dumps(dict(status=s, again=status(ws.loss_grad, x, t))))
""", tmp_path)
    assert out == dict(status=3, again=0)


def test_an_error_left_by_the_program_is_not_the_trainings(tmp_path):
    out = fakecuda.run(TRAIN + """
p = ctypes.c_void_p()
fake.cudaGetSymbolAddress(ctypes.byref(p), None)        # fails, and nobody asks for the error
print(json.dumps([status(ws.train, x, t, epochs=1, batch=2, lr=1e-3), status(ws.loss_grad, x, t)]))
""", tmp_path)
    assert out == [0, 0]
