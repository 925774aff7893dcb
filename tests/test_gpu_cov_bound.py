"""The eigenvalue bound of the covariances against FP64, relative to the bounded
result: each raw covariance (the same search without a bound) is clamped with
eigenvalues in FP64.  Clouds whose largest eigenvalues lie up to 1e6 times above
the bound while the small ones lie about its lower end (points along a cable
or a corridor), round ones whose eigenvalues nearly meet, and ordinary surfaces.
Tolerance: rounding the six entries to float is at most 2^-24 of the result's
Frobenius norm; 2^-23 leaves as much again for everything else."""
import numpy as np
import pytest

from helpers import soa
from paper_2606_10019_gb300 import datagen as D

pytestmark = pytest.mark.gpu


def _cloud(kind, n, rng):
    if kind == "surfaces":
        return D.make_corner_pair(n_src=n, n_tgt=n, frame=5).src_xyz
    if kind == "ball":
        return rng.normal(size=(n, 3))
    if kind == "pixels":      # equal steps along two axes: eigenvalues that meet
        a = np.arange(n)
        return np.c_[a % 64, a // 64, np.zeros(n)] * 0.05 + rng.normal(size=(n, 3)) * [0, 0, 1e-3]
    step, across = kind       # along a line that lies askew, with noise across it
    x = np.c_[step * (np.arange(n) + rng.uniform(-0.3, 0.3, n)), rng.normal(size=(n, 2)) * [across, 0.2 * across]]
    R = np.linalg.qr(np.random.default_rng(7).normal(size=(3, 3)))[0]
    return x @ R.T


@pytest.mark.parametrize("kind,n,eig,ratio", [
    ("surfaces", 4000, 0.01, 100.0), ("ball", 3000, 0.01, 100.0), ("ball", 3000, 1e3, 1e4), ("pixels", 4096, 0.09, 1e3),
    ((1.0, 0.05), 2000, 0.01, 100.0), ((3.0, 0.02), 2000, 0.01, 100.0), ((30.0, 0.05), 1500, 0.01, 100.0),
    ((30.0, 0.3), 1500, 0.09, 100.0), ((300.0, 0.1), 500, 0.01, 1e3), ((1e-12, 1e-13), 500, 1e-24, 100.0)])
def test_bound_matches_fp64(kind, n, eig, ratio):
    import torch
    from paper_2606_10019_gb300 import build as B
    from paper_2606_10019_gb300 import gcvo as G
    B.build()
    x = np.ascontiguousarray(_cloud(kind, n, np.random.default_rng(n)), dtype=np.float32)
    ctx = G.gcvo_create(0)
    out = []
    for e in (0.0, eig):
        c = torch.empty((6, n), device="cuda:0")
        G.gcvo_estimate_covariances(ctx, soa(x, "cuda:0"), G.kernel_params(knn=10, eig_max=e, eig_ratio=ratio), c)
        out.append(c.cpu().numpy().T.astype(np.float64)[:, [0, 1, 2, 1, 3, 4, 2, 4, 5]].reshape(-1, 3, 3))
    ctx.close()
    w, V = np.linalg.eigh(out[0])
    ref = np.einsum("nak,nk,nbk->nab", V, np.clip(w, eig / ratio, eig), V)
    norm = lambda m: np.linalg.norm(m, axis=(1, 2))
    err = norm(out[1] - ref) / norm(ref)
    assert err.max() <= 2.0 ** -23, err.max()
