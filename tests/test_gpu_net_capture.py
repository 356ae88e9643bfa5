"""Network calls in a caller's CUDA graph.  A captured call replays between direct ones, after the
weights have changed and after calls of other sizes, so nothing it needs may be left from a call
before it.  The expected values are those of a net of its own that makes direct calls only: the same
kernels, so equal bit for bit."""
import numpy as np
import pytest
import torch

from paper_2109_13628_gb300 import learned

pytestmark = pytest.mark.gpu

DILS = (1, 4, 2)


def weights(seed):
    n = learned.Net(in_channels=3, hidden=32, dilations=DILS, seed=seed)
    p = n.get()
    n.close()
    return p


def net_with(p):
    n = learned.Net(in_channels=3, hidden=32, dilations=DILS, seed=0)
    n.set(p)
    return n


def image(shape, seed):
    b, h, w = shape
    return torch.as_tensor(np.random.default_rng(seed).normal(size=(b, 3, h, w)).astype(np.float32), device="cuda")


def direct(p, x):
    n = net_with(p)
    y = torch.empty(x.shape[0], 1, *x.shape[2:], device="cuda")
    n.forward(x, y)
    y = y.clone()
    torch.cuda.synchronize()
    n.close()
    return y


def forward(n, x):
    y = torch.full((x.shape[0], 1, *x.shape[2:]), float("nan"), device="cuda")
    n.forward(x, y)
    return y


def capture(n, x):
    y = torch.full((x.shape[0], 1, *x.shape[2:]), float("nan"), device="cuda")
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        n.forward(x, y)
    return g, y


def test_replay_follows_the_weights():
    p, q = weights(1), weights(2)
    x = image((2, 37, 150), 3)
    n = net_with(p)
    forward(n, x)
    g, y = capture(n, x)
    g.replay()
    assert torch.equal(y, direct(p, x))
    n.set(q)
    g.replay()
    assert torch.equal(y, direct(q, x))
    t = torch.zeros_like(y)
    n.train_step(x, t, torch.ones_like(t), 0.01)
    g.replay()
    assert torch.equal(y, direct(n.get(), x)) and not torch.equal(y, direct(q, x))
    n.close()


def test_capture_without_replay_leaves_direct_calls_right():
    p, q = weights(1), weights(2)
    x, x2 = image((2, 37, 150), 3), image((1, 20, 140), 4)
    n = net_with(p)
    forward(n, x)
    n.set(q)
    g, y = capture(n, x)            # recorded, not run
    assert torch.equal(forward(n, x), direct(q, x))
    g2, y2 = capture(n, x2)
    assert torch.equal(forward(n, x2), direct(q, x2))
    g.replay()
    g2.replay()
    assert torch.equal(y, direct(q, x)) and torch.equal(y2, direct(q, x2))
    n.close()


# the second: fewer pixels, but more room in the padded buffers than the captured call had
@pytest.mark.parametrize("other", [(1, 60, 90), (1, 2500, 1), (3, 64, 200)])
def test_replay_between_calls_of_another_size(other):
    p = weights(5)
    x, x2 = image((2, 37, 150), 3), image(other, 6)
    n = net_with(p)
    forward(n, x)
    g, y = capture(n, x)
    for _ in range(2):
        assert torch.equal(forward(n, x2), direct(p, x2))
        g.replay()
        assert torch.equal(y, direct(p, x))
    n.close()


@pytest.mark.parametrize("shape", [(2, 37, 150), (1, 64, 64)])
def test_training_step_captured_after_inference_only(shape):
    """The buffers of a training step exist once a direct call of the size has run, whichever it was."""
    p = weights(7)
    x = image(shape, 8)
    t = torch.zeros(shape[0], 1, *shape[1:], device="cuda")
    m = torch.ones_like(t)
    n, ref = net_with(p), net_with(p)
    forward(n, x)
    ref.train_step(x, t, m, 0.01)
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        n.train_step(x, t, m, 0.01, want_loss=False)
    x2 = image((3, 90, 90), 9)
    assert torch.equal(forward(n, x2), direct(p, x2))      # larger buffers; the graph keeps its own
    g.replay()
    torch.cuda.synchronize()
    assert np.array_equal(n.get(), ref.get()) and not np.array_equal(n.get(), p)
    n.close()
    ref.close()
