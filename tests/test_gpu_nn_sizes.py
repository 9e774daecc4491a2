"""The proposal network's kernels at the batch sizes where their tiling changes:
one sample, ragged 8-sample clusters of the fully connected layers, the last size
of the 2-sample convolution blocks and the first of the 4-sample ones, the last
size of the clusters and the first of the 32-sample tiles, more
samples than blocks of the backward pass.  Against the FP64 oracle network with
the same BF16-rounded weights; tolerances as in test_gpu_nn.py (FP32 sums)."""
import numpy as np
import pytest

from test_gpu_nn import dev, make_inputs, make_params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def glt():
    import paper_2607_16897_gb300 as g
    return g


@pytest.fixture(scope="module")
def onn():
    from oracle import nn
    return nn


@pytest.mark.parametrize("B", [2, 9, 303, 304, 305, 2048, 2049])
def test_forward_sizes(glt, onn, B):
    import torch
    w = make_params(onn, 3)
    x, m, _ = make_inputs(B, 100 + B)
    net = glt.NN(B, w)
    y = torch.full((B + 1, 8), 7.0, device="cuda")
    net.forward(dev(x), dev(m), y, B)
    torch.cuda.synchronize()
    yo, _ = onn.forward(onn.unflatten(onn.to_bf16(w)), x.reshape(B, 1, 30, 40), m)
    y = y.cpu().numpy()
    assert np.abs(y[:B] - yo).max() <= 1e-4 * max(1.0, np.abs(yo).max())
    assert (y[B] == 7.0).all()          # nothing past the batch
    net.close()


@pytest.mark.parametrize("B", [1, 3, 63, 65, 149, 310])
def test_gradient_sizes(glt, onn, B):
    w = make_params(onn, 5)
    x, m, t = make_inputs(B, 200 + B)
    net = glt.NN(B, w)
    g, loss = net.gradient(dev(x), dev(m), dev(t), B)
    p = onn.unflatten(onn.to_bf16(w))
    y, cache = onn.forward(p, x.reshape(B, 1, 30, 40), m)
    go, _, _ = onn.backward(p, cache, y, t)
    assert abs(loss - onn.loss(y, t)) <= 1e-5 * onn.loss(y, t)
    gg = onn.unflatten(g.astype(np.float64))
    for name, _ in onn.SHAPES:
        rel = np.linalg.norm(gg[name] - go[name]) / np.linalg.norm(go[name])
        assert rel <= 1e-3, (B, name, rel)
    net.close()


def test_output_over_an_input(glt, onn):
    """y written over the motion input gives the same values (it is staged)."""
    import torch
    B = 40
    w = make_params(onn, 3)
    x, m, _ = make_inputs(B, 7)
    net = glt.NN(B, w)
    y = torch.zeros(B, 8, device="cuda")
    net.forward(dev(x), dev(m), y, B)
    buf = torch.zeros(B * 8, device="cuda")
    buf[:B * 6] = dev(m).reshape(-1)
    net.forward(dev(x), buf, buf, B)
    torch.cuda.synchronize()
    assert torch.equal(buf.reshape(B, 8), y)
    net.close()
