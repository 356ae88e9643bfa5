"""Inference of the learned guess's network on BF16 channel units (persistent tensor-core blocks, bulk
copies, four output rows per tile) against the numpy oracle that rounds every layer's input to BF16.
Inputs and weights are small integers, so every FP32 sum is exact whatever its order and the two
sides agree bit for bit: widths around the 128-pixel runs, heights around the row blocks of each
dilation, channel counts that leave groups of the MMA's K and columns of its N empty, several images, and
one net called with changing sizes (the zero borders of its buffers)."""
import numpy as np
import pytest
import torch

from oracle import net as onet
from paper_2109_13628_gb300 import learned
from tests.test_gpu_conv_tc import bf16_round, unpack

pytestmark = pytest.mark.gpu


def make(cin, hidden, dils, rng):
    net = learned.Net(in_channels=cin, hidden=hidden, dilations=dils, seed=1, tensor_cores=2)
    net.set(rng.integers(-1, 2, size=net.n).astype(np.float32))
    return net, unpack(net.get(), cin, hidden, len(dils))


def check(net, params, cin, dils, shape, rng):
    b, h, w = shape
    x = rng.integers(-3, 4, size=(b, cin, h, w)).astype(np.float32)
    y = torch.full((b, 1, h, w), float("nan"), dtype=torch.float32, device="cuda")
    net.forward(torch.as_tensor(x, device="cuda"), y)
    a = x.astype(np.float64)
    for li, ((wt, bias), d) in enumerate(zip(params, dils)):
        a = onet.conv2d(bf16_round(a).astype(np.float64), wt, bias, d)
        if li < len(dils) - 1:
            a = np.maximum(a, 0.0)
    assert np.abs(a).max() < 2 ** 24
    assert np.array_equal(y.cpu().numpy(), a.astype(np.float32))
    assert net.tensor_core_status() == (2, 0)


@pytest.mark.parametrize("cin,hidden,dils,shape", [
    (3, 32, (1, 1), (1, 1, 1)), (3, 32, (1, 2), (2, 4, 127)), (1, 8, (4, 1), (1, 15, 128)), (8, 9, (3, 1), (3, 13, 129)),
    (9, 17, (2, 5), (1, 41, 60)), (17, 24, (16, 1), (1, 65, 257)), (32, 32, (32, 1), (2, 33, 131)), (5, 1, (1,), (1, 7, 300))])
def test_units_forward_is_exact(cin, hidden, dils, shape):
    rng = np.random.default_rng(cin * 100 + hidden)
    net, params = make(cin, hidden, dils, rng)
    check(net, params, cin, dils, shape, rng)
    net.close()


def test_units_forward_with_changing_sizes():
    rng = np.random.default_rng(11)
    dils = (2, 8)
    net, params = make(3, 32, dils, rng)
    for shape in [(1, 40, 200), (2, 17, 90), (1, 40, 200), (1, 9, 260), (3, 5, 5)]:
        check(net, params, 3, dils, shape, rng)
    net.close()
