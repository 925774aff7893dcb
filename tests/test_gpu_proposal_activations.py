"""The proposal's backward pass recomputes the activations of layer 1 in the
forward's order of summation: an output whose sum is zero in that order, and
2^-24 with the bias added first, has no gradient."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
SHAPES = [(64, 4), (64,), (128, 64), (128,), (256, 128), (256,), (256, 512), (256,), (128, 256), (128,), (6, 128), (6,)]


@pytest.mark.parametrize("n", [2, 300])
def test_backward_sees_the_forwards_layer_1(n):
    import torch
    from paper_2606_10019_gb300 import build as B
    from paper_2606_10019_gb300 import gcvo as G
    B.build()
    W = [np.full(s, 0.01, np.float32) for s in SHAPES]
    W[0][:], W[1][:] = 0.0, 0.0
    W[0][0] = [2.0 ** -24, 0, 0, 1]      # x' 2^-24 + l - 1: 1 + x' 2^-24 rounds to 1 for x' < 1
    W[1][0] = -1.0
    W[0][1] = [0, 0, 0, 1]               # an ordinary output: l
    rng = np.random.default_rng(n)
    t = rng.normal(size=(1, 3, n)).astype(np.float32)
    c = t[0].astype(np.float64).mean(1)
    s = np.sqrt(((t[0] - c[:, None]) ** 2).sum(0).mean())
    z = (c[:, None] + s * rng.uniform(0.6, 0.9, (3, n)))[None].astype(np.float32)
    dev = lambda a: torch.from_numpy(a).to("cuda:0")
    ctx = G.gcvo_create(0)
    net = G.Proposal(ctx)
    net.set_params(np.concatenate([w.ravel() for w in W]))
    T = np.eye(4)
    T[:3, 3] = [0.3, -0.2, 0.1]
    _, grad = net.train_step(dev(z), dev(np.ones((1, n), np.float32)), dev(t), dev(np.zeros((1, n), np.float32)), T[None], 0.0,
                             want_grad=True)
    net.close()
    ctx.close()
    gW1, gb1 = grad[:256].reshape(64, 4), grad[256:320]
    assert gb1[1] != 0.0 and gW1[1, 3] != 0.0
    assert gb1[0] == 0.0 and not gW1[0].any()
