"""The convolutions' gradients are sums over every sample and position, which
the kernels take apart by blocks.  Their error against the FP64 oracle may not
exceed that of one block of 128 chains and a tree per parameter (geometric mean
over eight networks, relative to the layer's norm; measured on these inputs)."""
import numpy as np
import pytest

from test_gpu_nn import dev, make_inputs, make_params

pytestmark = pytest.mark.gpu

BOUNDS = {148: {"conv1.w": 2.203e-07, "conv2.w": 1.325e-07, "conv3.w": 1.108e-07, "conv3.b": 8.164e-08},
          256: {"conv1.w": 1.976e-07, "conv2.w": 1.089e-07, "conv3.w": 9.231e-08, "conv3.b": 7.144e-08}}


@pytest.mark.parametrize("B", sorted(BOUNDS))
def test_gradient_error_of_the_convolutions(B):
    import paper_2607_16897_gb300 as glt
    from oracle import nn as onn
    logs = {name: [] for name in BOUNDS[B]}
    for seed in range(8):
        w = make_params(onn, seed)
        x, m, t = make_inputs(B, 200 + seed)
        net = glt.NN(B, w)
        g, _ = net.gradient(dev(x), dev(m), dev(t), B)
        net.close()
        p = onn.unflatten(onn.to_bf16(w))
        y, cache = onn.forward(p, x.reshape(B, 1, 30, 40), m)
        go, _, _ = onn.backward(p, cache, y, t)
        gg = onn.unflatten(g.astype(np.float64))
        for name in logs:
            logs[name].append(np.log(np.linalg.norm(gg[name] - go[name]) / np.linalg.norm(go[name])))
    for name, bound in BOUNDS[B].items():
        assert np.exp(np.mean(logs[name])) <= bound, (name, np.exp(np.mean(logs[name])), bound)
