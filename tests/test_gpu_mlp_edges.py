"""The training kernel around its tiles (128 rows) and its grid (one tile per multiprocessor, then a
second one accumulated in tensor memory), and the update that takes the place of a gradient reduction,
an Adam step and a conversion: the next evaluation must see the new weights."""
import numpy as np
import pytest

from oracle import mlp as ref

pytestmark = pytest.mark.gpu


def _data(n):
    rng = np.random.default_rng(n)
    x = rng.uniform(-1, 1, size=(n, 2)).astype(np.float32)
    t = np.stack([np.sin(2 * x[:, 0]) * x[:, 1], np.cos(x[:, 1])], 1).astype(np.float32)
    m = (0.2 + rng.random((n, 2))).astype(np.float32)
    return x, t, m


@pytest.mark.parametrize("n", [1, 127, 128, 129, 152 * 128, 152 * 128 + 1])
def test_loss_gradient_and_step(n):
    from paper_2405_12964_gb300 import dwos
    p = ref.init_params(7) * 2.0
    x, t, m = _data(n)
    net = dwos.ControlVariateNet(params=p.astype(np.float32))
    loss, g = net.loss_grad(x, t, m)
    Lr, Gr, E, EL = ref.kernel_grad_bound(p, x.astype(np.float64), t, m)
    assert abs(float(loss[0]) - Lr) <= EL
    assert np.all(np.abs(g.cpu().numpy().astype(np.float64) - Gr) <= E)
    step = net.train_step(x, t, m, lr=1e-3)
    assert float(step[0]) == float(loss[0])      # the same kernel and sums
    # a network made from the stepped parameters has the same BF16 weights as the update left
    other = dwos.ControlVariateNet(params=net.params().cpu().numpy())
    for a, b in zip(net.eval(x), other.eval(x)):
        assert np.array_equal(a.cpu().numpy().view(np.uint32), b.cpu().numpy().view(np.uint32))
