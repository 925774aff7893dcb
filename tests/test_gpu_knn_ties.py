"""Which neighbours the covariances take where distances tie: the lower indices.
Points on a lattice of eighths, many of them copies, so that squared distances
and sums are exact in float; against brute force that sorts by (squared
distance, index).  The one rounding left is the division by knn - 1."""
import numpy as np
import pytest

from helpers import soa

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,span,knn", [(40, 1, 16), (3000, 16, 10), (3000, 4, 10), (9000, 40, 7), (70000, 60, 10)])
def test_ties_go_to_the_lower_index(n, span, knn):
    import torch
    from paper_2606_10019_gb300 import build as B
    from paper_2606_10019_gb300 import gcvo as G
    B.build()
    k = np.random.default_rng(n + span).integers(-span, span + 1, (n, 3))
    x = (k / 8.0).astype(np.float32)
    ctx = G.gcvo_create(0)
    cov = torch.empty((6, n), device="cuda:0")
    G.gcvo_estimate_covariances(ctx, soa(x, "cuda:0"), G.kernel_params(knn=knn, eig_max=0.0), cov)
    ctx.close()
    X = torch.from_numpy(k).to("cuda:0")
    order = torch.arange(n, device="cuda:0")
    at = torch.from_numpy(np.random.default_rng(1).permutation(n)[:2000]).to("cuda:0")
    for a in at.split(500):
        d = X[None] - X[a][:, None]
        key = (d * d).sum(2) * n + order              # whole numbers: (squared distance, index)
        y = torch.gather(d, 1, key.topk(knn, largest=False).indices[:, :, None].expand(-1, -1, 3)).double() / 8.0
        S = torch.einsum("nka,nkb->nab", y, y)[:, [0, 0, 0, 1, 1, 2], [0, 1, 2, 1, 2, 2]] / (knn - 1)
        got = cov[:, a].T.double()
        assert float(((got - S).abs() - 2.0 ** -22 * S.abs()).max()) <= 0.0
