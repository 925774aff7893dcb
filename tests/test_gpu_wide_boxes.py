"""Sub-tiles whose box spans much of the scene, where the pair pass's second list
saves too little to count apart: points in no order (gcvo_eval_static takes them
as they come) and sparse clouds, whose sub-tiles of 32 reach far, against the
sorted evaluation of the same points and against sub-tiles of 4; counts equal.
Tolerance: the repository's 1e-5 on f, g and H."""
import numpy as np
import pytest

from helpers import soa
from paper_2606_10019_gb300 import datagen as D
from test_gpu_parity import TOL, env  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,mixed", [(5, False), (700, True), (6000, False), (6000, True)])
def test_points_in_no_order(env, n, mixed):
    import torch
    O, G, ctx, dev = env
    rng = np.random.default_rng(n)
    p = D.make_corner_pair(n_src=max(n, 10), n_tgt=4000, frame=n)
    kp = G.kernel_params(eig_max=0.01)
    src = p.src_xyz[rng.permutation(len(p.src_xyz))[:n]]
    xyz = [soa(p.tgt_xyz, dev), soa(src, dev)]
    cov = [torch.empty((6, x.shape[1]), device=dev) for x in xyz]
    G.gcvo_estimate_covariances(ctx, xyz[0], kp, cov[0])
    cov[1][:] = torch.tensor([1e-4, 0, 0, 2e-4, 0, 1.5e-4], device=dev)[:, None]
    if mixed:     # some chunks near enough to their box for two lists
        cov[0][:, : 2000] *= 0.05
    f = [torch.rand((1, x.shape[1]), device=dev) for x in xyz]
    grid = G.gcvo_build_grid(ctx, xyz[0], cov[0], f[0], kp)
    T = D.rigid(np.eye(3), np.array([0.01, -0.02, 0.015]))
    out = []
    try:
        for sched in (4 | 1 << 8, 32 | 3 << 8):
            G.gcvo_pair_schedule(ctx, sched)
            out.append(G.gcvo_eval(ctx, grid, xyz[1], cov[1], f[1], T))
    finally:
        G.gcvo_pair_schedule(ctx, 0)
    fs, gs, Hs = G.gcvo_eval_static(grid, xyz[1], cov[1], f[1], T)
    grid.close()
    a, b = out
    assert (a.n_pairs, a.n_kept) == (b.n_pairs, b.n_kept) and (n < 100 or a.n_kept > 0)
    scale = np.abs(a.H).max()
    for ff, gg, HH in ((b.f, b.g, b.H), (fs, gs, Hs)):
        assert abs(ff - a.f) <= TOL * abs(a.f)
        assert np.abs(gg - a.g).max() <= TOL * max(np.abs(a.g).max(), np.sqrt(scale * abs(a.f)))
        assert np.linalg.norm(HH - a.H) <= TOL * np.linalg.norm(a.H)
