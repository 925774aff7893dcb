"""The register loop of G-CVO-2 as one cooperative kernel against the graph of
separate kernels (which runs while profiling is on): the same poses, logs and
iteration counts bit for bit, for one problem and for batches in which the
problems stop at different iterations, run out of iterations or fail, and a
loop longer than one launch of the kernel."""
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


def _problem(G, ctx, dev, n, frame, fd=1, **kw):
    import torch
    p = D.make_corner_pair(n_src=n, n_tgt=max(10, int(0.9 * n)), frame=frame)
    rng = np.random.default_rng(frame)
    kp = G.kernel_params(eig_max=0.01, feat_dim=fd, **kw)
    xyz = [soa(p.tgt_xyz, dev), soa(p.src_xyz, dev)]
    cov = [torch.empty((6, x.shape[1]), device=dev) for x in xyz]
    for x, c in zip(xyz, cov):
        G.gcvo_estimate_covariances(ctx, x, kp, c)
    f = [soa(rng.uniform(0.1, 1, (x.shape[1], fd)), dev) for x in xyz]
    return G.gcvo_build_grid(ctx, xyz[0], cov[0], f[0], kp), xyz[1], cov[1], f[1], np.eye(4)


def _both(G, ctx, call):
    a = call()
    G.gcvo_profile_enable(ctx, True)
    b = call()
    G.gcvo_profile_enable(ctx, False)
    return a, b


@pytest.mark.parametrize("n,fd,sched,kw", [
    (12, 1, 8, {}), (333, 3, 16, {}), (2000, 1, 4, {}), (2000, 7, 32, {}), (9000, 1, 8, {}),
    (1500, 1, 8, dict(kernel_mode=1, iso_ell=0.08)), (400, 5, 4, dict(cutoff=0.0))])
def test_one_problem(env, n, fd, sched, kw):
    G, ctx, dev = env
    prob = _problem(G, ctx, dev, n, 3, fd, **kw)
    sp = G.solver_params(k_max=37, eps_tol=1e-7)
    try:
        G.gcvo_pair_schedule(ctx, sched)
        a, b = _both(G, ctx, lambda: G.gcvo_register(ctx, *prob, sp))
    finally:
        G.gcvo_pair_schedule(ctx, 0)
    assert a[2] == b[2] and a[3] == b[3] and np.array_equal(a[0], b[0])
    assert a[1].tobytes() == b[1].tobytes()


def test_batch_and_long_loop(env):
    G, ctx, dev = env
    probs = [_problem(G, ctx, dev, n, f) for f, n in enumerate((1500, 40, 700, 5000, 15, 2500))]
    far = list(probs[2])
    far[4] = D.rigid(np.eye(3), np.array([50.0, 0.0, 0.0]))      # no overlap: fails at once
    probs.append(tuple(far))
    try:
        G.gcvo_pair_schedule(ctx, 8)
        for k_max, eps in ((60, 1e-6), (6, 1e-12), (1, 1e-6), (1100, 0.0)):
            sp = G.solver_params(k_max=k_max, eps_tol=eps)
            a, b = _both(G, ctx, lambda: G.gcvo_register_batched(ctx, probs, sp, want_log=True))
            assert np.array_equal(a[0], b[0]) and np.array_equal(a[2], b[2]) and np.array_equal(a[3], b[3])
            for x, y in zip(a[1], b[1]):
                assert x.tobytes() == y.tobytes()
            assert a[3][-1] == G.GCVO_ERR_NO_OVERLAP and a[2][:-1].max() <= k_max
            if eps == 0.0:
                assert a[2][:-1].max() == k_max
    finally:
        G.gcvo_pair_schedule(ctx, 0)


def test_large_sets_replay_the_graphs(env):
    """More than 2^39 pairs in all (copies of one problem): kernels of their own, and the same poses."""
    G, ctx, dev = env
    prob = _problem(G, ctx, dev, 60000, 3)
    copies = int(2.0 ** 39 // (60000 * 54000)) + 1
    sp = G.solver_params(k_max=3, eps_tol=1e-12)
    try:
        G.gcvo_pair_schedule(ctx, 8)
        one = G.gcvo_register(ctx, *prob, sp)
        many = G.gcvo_register_batched(ctx, [prob] * copies, sp)
    finally:
        G.gcvo_pair_schedule(ctx, 0)
    assert all(np.array_equal(T, one[0]) for T in many[0])
    assert set(many[2]) == {one[2]} and set(many[3]) == {one[3]}
