"""The weight-gradient kernel of the learned guess's network (register tiles of 8 x 4 channels per
lane, strips of 64 pixels) against the numpy oracle: widths around the strip length, channel counts
around the tile sizes (where lanes split the pixels instead), dilations up to the largest, and
reproducibility (the sums have a fixed order)."""
import numpy as np
import pytest
import torch

from oracle import net as onet
from paper_2109_13628_gb300 import learned
from tests.test_gpu_net import bf16_round, unpack

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cin,hidden,batch,h,w,d", [
    (1, 1, 1, 1, 1, 1), (3, 32, 2, 5, 63, 1), (3, 32, 1, 9, 64, 16), (4, 8, 3, 7, 65, 2), (5, 9, 1, 33, 40, 32),
    (8, 16, 1, 6, 129, 3), (17, 17, 2, 11, 30, 5), (32, 32, 1, 40, 191, 8)])
def test_weight_gradients_match_oracle(cin, hidden, batch, h, w, d):
    dev = torch.device("cuda", 0)
    dils = (d, 1)
    net = learned.Net(in_channels=cin, hidden=hidden, dilations=dils, seed=3, tensor_cores=0)
    rng = np.random.default_rng(cin + 100 * hidden + w)
    net.set((0.3 * rng.normal(size=net.n)).astype(np.float32))
    params = [(bf16_round(a).astype(np.float64), b) for a, b in unpack(net.get(), cin, hidden, 2)]
    x = rng.normal(size=(batch, cin, h, w)).astype(np.float32)
    dy = rng.normal(size=(batch, 1, h, w)).astype(np.float32)
    g = net.backward(torch.as_tensor(x, device=dev), torch.as_tensor(dy, device=dev))
    g2 = net.backward(torch.as_tensor(x, device=dev), torch.as_tensor(dy, device=dev))
    net.close()
    acts = onet.forward(params, list(dils), x.astype(np.float64))
    gx, gw1, gb1 = onet.conv2d_backward(acts[1], params[1][0], 1, dy.astype(np.float64))
    _, gw0, gb0 = onet.conv2d_backward(acts[0], params[0][0], d, gx * (acts[1] > 0))
    ref = np.concatenate([gw0.ravel(), gb0.ravel(), gw1.ravel(), gb1.ravel()])
    # FP32 products and sums of n = batch h w terms: rounding grows like sqrt(n) 2^-24 of the terms'
    # norm, which is at most n times the largest term; 1e-4 of the largest gradient covers n = 1e4 with
    # two orders to spare
    assert np.abs(g - ref).max() <= 1e-4 * max(np.abs(ref).max(), 1e-3)
    assert np.array_equal(g, g2)
