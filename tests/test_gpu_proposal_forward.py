"""The proposal's forward pass at the edges of its tiles (128 points of a
cloud) and of its split over blocks (several clouds per block, one cloud over
several blocks): twists against the FP64 oracle with the same BF16 weights,
relative error <= 1e-2 (BF16 layer inputs), the bound of the full-size test."""
import numpy as np
import pytest

from test_proposal_gpu import _oracle_batch, _pairs, _to_dev, bf16, penv  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,n", [(1, 1), (2, 127), (1, 128), (5, 129), (77, 100), (160, 130), (3, 5000), (1, 20001)])
def test_twists_match_oracle(penv, B, n):  # noqa: F811
    PR, G, ctx, dev = penv
    p = PR.init_params(8)
    rng = np.random.default_rng(B * n)
    for k in p:
        if k[0] in "bc":
            p[k] = rng.normal(scale=0.05, size=p[k].shape)
    net = G.Proposal(ctx)
    net.set_params(PR.flat(p).astype(np.float32))
    pairs = _pairs(min(B, 8), n, seed=6)
    pairs = [pairs[b % len(pairs)] for b in range(B)]
    tw, _ = net.infer(*_to_dev(pairs, dev))
    net.close()
    pq = {k: (bf16(v) if k[0] in "WH" else v.astype(np.float32).astype(np.float64)) for k, v in p.items()}
    batch, _ = _oracle_batch(PR, pairs[:8])
    out, _ = PR.forward(pq, batch)
    assert np.isfinite(tw).all()
    m = len(out)
    assert np.abs(tw[:m] - out).max() <= 1e-2 * np.abs(out).max()
    # the same pair gives the same twist wherever it sits in the batch
    for b in range(B):
        assert np.array_equal(tw[b], tw[b % m])
