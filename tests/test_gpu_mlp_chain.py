"""The one-launch chain of the surrogate's row products at its edges: a single row, a tile's
last and first rows, the largest batch in 32-row tiles on 152 SMs (4864 rows) and the first in
64-row tiles, several tiles a CTA with a ragged end.  Bounds are those of test_gpu_mlp:
C_BOUND BF16 scales an entry."""
import numpy as np
import pytest

from oracle import mlp as O
from tests.test_gpu_mlp import C_BOUND, _scales, _setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1, 127, 129, 4864, 4865, 20011])
def test_chain_entrywise(cuda, B):
    net, p, x, t, dx, dt = _setup(cuda, B)
    y = net.forward(dx).cpu().numpy().astype(np.float64)
    _, g = net.loss_grad(dx, dt)
    assert net.tcgen05
    y_ref, sy, g_ref, sg = _scales(p, x.astype(np.float64), t.astype(np.float64))
    assert (np.abs(y - y_ref) / sy).max() <= C_BOUND
    assert (np.abs(g.cpu().numpy() - g_ref) / (sg + 1e-300)).max() <= C_BOUND


def test_rows_do_not_depend_on_the_launch(cuda):
    """A row's product takes the same operations in tiles of 32 rows as of 64."""
    net, p, x, t, dx, dt = _setup(cuda, 4992)
    whole = net.forward(dx)
    for B in (1, 130, 4864):
        assert np.array_equal(net.forward(dx[:B].contiguous()).cpu().numpy(),
                              whole[:B].cpu().numpy())


def test_loss_of_successive_calls(cuda):
    """Each call's squared-error sum starts from zero, whatever ran before it.  The sum of
    1.3e6 non-negative FP64 terms in another order: relative difference below 1e-9."""
    net, p, x, t, dx, dt = _setup(cuda, 5000)
    small, st = dx[:300].contiguous(), dt[:300].contiguous()
    a, _ = net.loss_grad(small, st)
    b, _ = net.loss_grad(dx, dt)
    net.tcgen05 = False
    c, _ = net.loss_grad(small, st)
    net.tcgen05 = True
    for _ in range(2):
        net.forward(dx)
        assert net.loss_grad(small, st)[0] == pytest.approx(a, rel=1e-9)
        net.train_step(small, st, 1e-12)  # (moves the parameters by less than their last bit)
        assert net.loss_grad(dx, dt)[0] == pytest.approx(b, rel=1e-6)
    assert c == pytest.approx(a, rel=2e-2)
