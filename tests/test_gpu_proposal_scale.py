"""The proposal's normalisation far from the origin: centroid and RMS radius of
the target as the proposed poses use them, against FP64.  With all weights zero
and a bias of the last layer the twist is that bias, so the pose's translation
gives the radius and, for a half turn, the centroid.  Both are float values:
within a float's rounding (2^-24) of the FP64 ones, with 1e-9 for what comes
before and after the rounding."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("offset,size,n", [(0.0, 1.0, 257), (100.0, 1.0, 4096), (1e4, 1.0, 1000), (1e5, 3.0, 4095), (-3e6, 40.0, 513),
                                           (5.0, 1e-3, 64), (0.0, 1e6, 1)])
def test_radius_and_centroid(offset, size, n):
    import torch
    from paper_2606_10019_gb300 import build as B
    from paper_2606_10019_gb300 import gcvo as G
    B.build()
    rng = np.random.default_rng(n)
    t = (offset * np.array([1.0, -0.7, 0.1])[None, :, None] + size * rng.normal(size=(3, 3, n))).astype(np.float32)
    x = t.astype(np.float64)
    c = x.mean(2)
    s = np.sqrt(((x - c[:, :, None]) ** 2).sum(1).mean(1)) + 1e-6
    dev = lambda a: torch.from_numpy(a).to("cuda:0")
    ctx = G.gcvo_create(0)
    net = G.Proposal(ctx)

    def pose(twist):
        w = np.zeros(net.n_params, np.float32)
        w[-6:] = twist
        net.set_params(w)
        f = dev(np.zeros((3, n), np.float32))
        return net.infer(dev(t), f, dev(t), f)[1]

    radius = pose([0, 0, 0, 2.0 ** 20, 0, 0])[:, 0, 3] / 2.0 ** 20      # far above the rounding of c + v s - c in FP64
    half = pose([np.float32(np.pi), 0, 0, 0, 0, 0])[:, 1:3, 3] / 2.0      # (I - R) c / 2 = c beside the axis
    net.close()
    ctx.close()
    assert np.abs(radius / s - 1.0).max() <= 2.0 ** -24 + 1e-9
    tilt = 1e-7 * np.abs(c[:, 1:]).max(1, keepdims=True)                  # pi as a float turns c by 9e-8
    assert np.all(np.abs(half - c[:, 1:]) <= (2.0 ** -24 + 1e-9) * np.abs(c[:, 1:]) + tilt)
