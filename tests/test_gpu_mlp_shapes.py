"""Network kernels at widths and batches off their tile sizes (32 and 64
outputs, depth 64 per stage, rows padded to 8), forward and gradients against
the FP64 reference with the bounds of test_gpu_warmstart."""
import numpy as np
import pytest

import paper_2010_01847_gb300 as plbm
from oracle import mlp as omlp

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from test_gpu_warmstart import _grad_magnitudes, _rounded_params, bf16  # noqa: E402


@pytest.mark.parametrize("widths,batch", [
    ([1, 1], 1),                       # a single weight
    ([5, 7, 33, 9], 31),               # no width a multiple of 8
    ([3, 65, 31, 2], 97),
    ([20, 600, 40], 520),              # depth beyond the stages in flight
    ([3, 1000, 20], 1301),             # 64 x 64 tiles
])
def test_odd_shapes_match_oracle(widths, batch):
    net = plbm.Mlp(widths, max_batch=batch)
    net.init_params(seed=4)
    p = net.params()
    rng = np.random.default_rng(6)
    x = rng.uniform(-1, 1, (batch, widths[0])).astype(np.float32)
    t = rng.normal(0, 1, (batch, widths[-1])).astype(np.float32)
    rp = _rounded_params(net, p)
    y = net.forward(x).cpu().numpy()
    ref, _ = omlp.forward(rp, widths, bf16(x), hidden_round=bf16)
    assert np.abs(y - ref).max() <= 1e-2 * np.abs(ref).max()
    loss, g = net.loss_grad(x, t)
    ref_loss, ref_g = omlp.loss_grad(rp, widths, bf16(x), t, hidden_round=bf16)
    assert loss == pytest.approx(ref_loss, rel=1e-2)
    m = _grad_magnitudes(rp, widths, bf16(x), t)
    bound = len(widths) * 2.0 ** -8 * m + 1e-6 * np.abs(ref_g).max()
    assert (np.abs(g - ref_g) / bound).max() <= 1.0


def test_minibatch_larger_than_the_set_repeats_its_rows():
    """batch > n takes the rows in order, again from the first after the last:
    the same steps as on a set that holds them so (the loop read rows past the
    set's end before)."""
    widths = [3, 16, 24]
    rng = np.random.default_rng(8)
    x = rng.uniform(-1, 1, (40, 3)).astype(np.float32)
    t = rng.normal(0, 1, (40, 24)).astype(np.float32)
    rows = np.arange(100) % 40
    out = []
    for xs, ts in ((x, t), (x[rows], t[rows])):
        net = plbm.Mlp(widths, max_batch=100)
        net.init_params(seed=2)
        loss = net.train(xs, ts, steps=12, batch=100, lr=2e-3, lr_final=1e-3, seed=5)
        out.append((loss, net.params()))
    np.testing.assert_array_equal(out[0][0], out[1][0])
    np.testing.assert_array_equal(out[0][1], out[1][1])
