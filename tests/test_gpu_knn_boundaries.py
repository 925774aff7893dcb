"""Points whose neighbours in Morton order lie far away: a few of them alone
behind the largest cells' boundary, beside a dense cloud on the other side.  The
search starts from smaller cells there; against brute force in FP64."""
import numpy as np
import pytest

from helpers import soa
from test_gpu_knn_sizes import COV_TOL, _reference

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,alone,eig", [(20000, 1, 0.01), (20000, 4, 0.01), (30000, 9, 0.0), (66000, 4, 0.01), (66000, 12, 0.0)])
def test_points_alone_behind_a_boundary(n, alone, eig):
    import torch
    from paper_2606_10019_gb300 import build as B
    from paper_2606_10019_gb300 import gcvo as G
    B.build()
    rng = np.random.default_rng(n + alone)
    x = np.c_[rng.uniform(0, 2.0, (n, 2)), 0.01 * rng.normal(size=n)]
    # the longest axis runs to 2.05: some voxels beyond a power of two, with few points
    x[:alone] = np.c_[rng.uniform(2.0, 2.05, alone), rng.uniform(0, 2.0, alone), 0.01 * rng.normal(size=alone)]
    x = np.ascontiguousarray(rng.permutation(x), dtype=np.float32)
    ctx = G.gcvo_create(0)
    cov = torch.empty((6, n), device="cuda:0")
    G.gcvo_estimate_covariances(ctx, soa(x, "cuda:0"), G.kernel_params(knn=10, eig_max=eig, eig_ratio=100.0), cov)
    ctx.close()
    got = cov.cpu().numpy().T.astype(np.float64)[:, [0, 1, 2, 1, 3, 4, 2, 4, 5]].reshape(-1, 3, 3)
    ref, raw, gap = _reference(x, 10, eig)
    norm = lambda m: np.linalg.norm(m, axis=(1, 2))
    ok = gap > 1e-5
    assert ok.mean() > 0.9
    assert (norm(got - ref) / np.maximum(norm(ref), norm(raw)))[ok].max() <= COV_TOL
