"""lb_ws_train when a CUDA call fails (fake runtime, no GPU): the parameters stay as they were."""
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
