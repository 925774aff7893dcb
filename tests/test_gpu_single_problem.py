"""The one-launch preparation of a single problem (up to 65,536 source points)
against the batched preparation: the same two iterations bit for bit -- f, g,
step, pose, pair counts -- at the edges of the cluster's tiles, every cut of
the work items, every number of feature channels, both kernels and the dense
objective; and a non-finite input ends a registration with its status."""
import numpy as np
import pytest

from helpers import soa
from paper_2606_10019_gb300 import datagen as D

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    from paper_2606_10019_gb300 import build as B
    from paper_2606_10019_gb300 import gcvo as G
    B.build()
    ctx = G.gcvo_create(0)
    yield G, ctx, torch.device("cuda:0")
    ctx.close()


def _problem(G, ctx, dev, n, fd, **kw):
    pair = D.make_corner_pair(n_src=max(n, 10), n_tgt=900, frame=n)
    rng = np.random.default_rng(n + fd)
    kp = G.kernel_params(eig_max=0.01, feat_dim=fd, **kw)
    tx, sx = soa(pair.tgt_xyz, dev), soa(pair.src_xyz[:n], dev)
    import torch
    cov = []
    for x in (tx, soa(pair.src_xyz, dev)):
        c = torch.empty((6, x.shape[1]), device=dev)
        G.gcvo_estimate_covariances(ctx, x, kp, c)
        cov.append(c)
    f = lambda m: soa(rng.uniform(0.1, 1, (m, fd)), dev)
    grid = G.gcvo_build_grid(ctx, tx, cov[0], f(900), kp)
    return grid, (sx, cov[1][:, :n].contiguous(), f(n))


@pytest.mark.parametrize("n,fd,sched,kw", [
    (1, 1, 4 | 1 << 8, {}), (31, 3, 8 | 1 << 8, {}), (1024, 1, 8 | 2 << 8, {}), (1025, 7, 16 | 2 << 8, {}),
    (2049, 1, 32 | 3 << 8, {}), (5000, 5, 4 | 2 << 8, dict(kernel_mode=1, iso_ell=0.08)),
    (16385, 1, 8 | 3 << 8, {}), (40000, 3, 16 | 3 << 8, {}), (65536, 1, 32 | 2 << 8, {}),
    (700, 1, 8 | 2 << 8, dict(cutoff=0.0)), (3000, 1, 8 | 1 << 8, dict(sigma2=2.5))])
def test_single_equals_batched(env, n, fd, sched, kw):
    G, ctx, dev = env
    grid, src = _problem(G, ctx, dev, n, fd, **kw)
    sp = G.solver_params(k_max=2, eps_tol=0.0)
    T0 = D.rigid(np.eye(3), np.array([0.01, -0.02, 0.015]))
    try:
        G.gcvo_pair_schedule(ctx, sched)
        T, log, _, _ = G.gcvo_register(ctx, grid, *src, T0, sp)
        Tb, logs, _, _ = G.gcvo_register_batched(ctx, [(grid, *src, T0)] * 2, sp, want_log=True)
        r = G.gcvo_eval(ctx, grid, *src, T0)
    finally:
        G.gcvo_pair_schedule(ctx, 0)
    for k in range(2):
        assert np.array_equal(T, Tb[k])
        for name in ("f", "g", "xi", "T", "n_pairs", "n_kept"):
            assert np.array_equal(log[name], logs[k][name]), name
    assert r.f == log[0]["f"] and np.array_equal(r.g, log[0]["g"]) and r.n_pairs == log[0]["n_pairs"]
    grid.close()


@pytest.mark.parametrize("which", [0, 1])
def test_non_finite_input_ends_a_registration(env, which):
    G, ctx, dev = env
    grid, src = _problem(G, ctx, dev, 2500, 1)
    src = [a.clone() for a in src]
    src[which][1, 1234] = float("nan")
    with pytest.raises(G.GcvoError) as e:
        G.gcvo_register(ctx, grid, *src, np.eye(4), G.solver_params(k_max=100000))
    assert e.value.status == G.GCVO_ERR_NONFINITE
    with pytest.raises(G.GcvoError) as e:
        G.gcvo_eval(ctx, grid, *src, np.eye(4))
    assert e.value.status == G.GCVO_ERR_NONFINITE
    grid.close()
