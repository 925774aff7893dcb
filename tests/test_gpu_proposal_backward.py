"""The proposal's backward pass at the edges of its work split (units of 64
channels of one cloud, one or two per block up to several), against the FP64
oracle: gradient cosine >= 0.999, the bound of the full-size test (BF16
activations), per parameter tensor."""
import numpy as np
import pytest

from test_proposal_gpu import _oracle_batch, _pairs, _to_dev, bf16, penv  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,n", [(1, 1), (1, 17), (3, 200), (41, 129)])
def test_gradient_of_small_and_ragged_batches(penv, B, n):  # noqa: F811
    PR, G, ctx, dev = penv
    p = PR.init_params(5)
    rng = np.random.default_rng(9)
    for k in p:
        if k[0] in "bc":
            p[k] = rng.normal(scale=0.05, size=p[k].shape)
    net = G.Proposal(ctx)
    net.set_params(PR.flat(p).astype(np.float32))
    pairs = _pairs(B, n, seed=4)
    _, grad = net.train_step(*_to_dev(pairs, dev), np.stack([q[4] for q in pairs]), lr=0.0, want_grad=True)
    net.close()
    pq = {k: (bf16(v) if k[0] in "WH" else v.astype(np.float32).astype(np.float64)) for k, v in p.items()}
    batch, labels = _oracle_batch(PR, pairs)
    _, g_o = PR.loss_and_grad(pq, batch, labels)
    assert np.all(np.isfinite(grad))
    got = PR.unflat(grad.astype(np.float64))
    for k, ref in g_o.items():
        a, b = np.ravel(got[k]), np.ravel(ref)
        if np.linalg.norm(b) == 0.0:
            assert np.linalg.norm(a) == 0.0
        else:
            assert a @ b / (np.linalg.norm(a) * np.linalg.norm(b)) >= 0.999, k
