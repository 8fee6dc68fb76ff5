"""The loss of a training call is that of its own batch, whatever ran, was captured or was
replayed before it: a training step without a loss can be captured into a CUDA graph, which
then runs between direct calls, any number of times or never."""
import pytest

from tests.test_gpu_mlp import _setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("replays", [0, 1, 3])
@pytest.mark.parametrize("before", [0, 1, 2])
def test_loss_beside_a_captured_step(cuda, before, replays):
    net, p, x, t, dx, dt = _setup(cuda, 300)
    # steps that move the parameters by less than their last bit: the loss stays `want`, the
    # sum of 76 800 non-negative terms (FP32 in groups of 16, then FP64) in whatever order
    want = net.loss_grad(dx, dt)[0]
    s = cuda.cuda.Stream()
    from paper_1906_09530_gb300 import Mlp
    net = Mlp(max_batch=512, stream=s)
    net.set_params(p)
    for _ in range(before):
        assert net.loss_grad(dx, dt)[0] == pytest.approx(want, rel=1e-9)
    cuda.cuda.synchronize()
    g = cuda.cuda.CUDAGraph()
    with cuda.cuda.graph(g, stream=s):
        net.train_step(dx, dt, 1e-12)
    for _ in range(replays):
        g.replay()
    cuda.cuda.synchronize()
    for _ in range(3):  # one and two direct calls between replays
        for _ in range(2):
            assert net.loss_grad(dx, dt)[0] == pytest.approx(want, rel=1e-9)
            g.replay()
            cuda.cuda.synchronize()
        assert net.train_step(dx, dt, 1e-12, want_loss=True) == pytest.approx(want, rel=1e-9)


def test_loss_has_one_order_of_summation(cuda):
    """The same call gives the same loss bit for bit: its partial sums are added in a fixed
    order."""
    net, p, x, t, dx, dt = _setup(cuda, 5000)
    first, _ = net.loss_grad(dx, dt)
    assert all(net.loss_grad(dx, dt)[0] == first for _ in range(20))
