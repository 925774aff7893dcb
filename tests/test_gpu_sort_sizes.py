"""Source sorts at the edges of the cluster sort's tiles (1024 keys per block,
1, 2 or 4 per thread, 16 blocks) and of its range (65,536 keys): an evaluation
sums every source point once, so f and g against a direct FP64 sum over all
pairs show a lost, doubled or misplaced point.  Tolerance: the 1e-5 of every
evaluation."""
import numpy as np
import pytest

from helpers import TOL, rel_f, soa

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 33, 1023, 1024, 1025, 2048, 2049, 8193, 16384, 16385, 32768, 32769, 65536, 65537])
@pytest.mark.parametrize("problems", [1, 3])
def test_every_source_point_counts_once(n, problems):
    import torch
    from paper_2606_10019_gb300 import build as B
    from paper_2606_10019_gb300 import gcvo as G
    B.build()
    dev = torch.device("cuda:0")
    ell, rng = 0.2, np.random.default_rng(n)
    x = rng.uniform(0, 2, size=(257, 3)).astype(np.float32)
    lx = rng.uniform(0.2, 1, size=(257, 1)).astype(np.float32)
    z = rng.uniform(0, 2, size=(n, 3)).astype(np.float32)
    lz = rng.uniform(0.2, 1, size=(n, 1)).astype(np.float32)
    ctx = G.gcvo_create(0)
    kp = G.kernel_params(kernel_mode=1, iso_ell=ell)
    grid = G.gcvo_build_grid(ctx, soa(x, dev), None, soa(lx, dev), kp)
    X, Z = torch.from_numpy(x).to(dev).double(), torch.from_numpy(z).to(dev).double()
    r = X[:, None] - Z[None]
    d2 = (r ** 2).sum(2) / ell ** 2
    w = torch.from_numpy(lx).to(dev).double() * torch.from_numpy(lz).to(dev).double().T * torch.exp(-0.5 * d2) * (d2 <= 9.0)
    u = (w[..., None] * r).sum(0) / ell ** 2
    f = float(w.sum())
    g = -torch.cat([torch.linalg.cross(Z, u).sum(0), u.sum(0)]).cpu().numpy()
    scale = float((w * torch.linalg.norm(r, dim=2)).sum()) / ell ** 2 * 2.0     # of the sums g cancels from
    if problems == 1:
        e = G.gcvo_eval(ctx, grid, soa(z, dev), None, soa(lz, dev), np.eye(4))
        got = [(e.f, e.g)]
    else:
        sp = G.solver_params(k_max=1)
        probs = [(grid, soa(z[:m], dev), None, soa(lz[:m], dev), np.eye(4)) for m in (max(1, n // 2), n, max(1, n // 3))]
        _, logs, _, _ = G.gcvo_register_batched(ctx, probs, sp, want_log=True)
        got = [(logs[1][0]["f"], logs[1][0]["g"])]
    for fg, gg in got:
        assert rel_f(fg, f) <= TOL
        assert np.abs(gg - g).max() <= TOL * scale
    grid.close()
    ctx.close()
