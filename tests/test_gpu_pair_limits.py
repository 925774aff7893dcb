"""The limits by which the pair pass leaves targets out of its evaluated list
must not leave out a pair that passes the cutoff: pairs laid just inside it
along an axis, in sub-tiles with two lists (one target with a large covariance
sets rho for all)."""
from types import SimpleNamespace

import numpy as np
import pytest

from helpers import Case, rel_f_near
from paper_2606_10019_gb300 import datagen as D
from test_gpu_parity import TOL, env  # noqa: F401

pytestmark = pytest.mark.gpu
SIX = ([0, 0, 0, 1, 1, 2], [0, 1, 2, 1, 2, 2])


def _case(O, G, ctx, dev, tx, tc, sx, sc):
    rng = np.random.default_rng(1)
    f = lambda n: rng.uniform(0.5, 1, (n, 1)).astype(np.float32)
    pair = SimpleNamespace(tgt_xyz=tx.astype(np.float32), src_xyz=sx.astype(np.float32), tgt_feat=f(len(tx)),
                           src_feat=f(len(sx)))
    case = Case(O, pair, O.KernelParams(cutoff=3.0), iso=True)
    case.iso, case.tc, case.sc = False, tc, sc
    case.prob = O.Problem.make(pair.tgt_xyz, tc, pair.tgt_feat, pair.src_xyz, sc, pair.src_feat)
    return case.gpu(G, ctx, dev, G.kernel_params(eig_max=0.01))


@pytest.mark.parametrize("sigma,half", [(5e-5, 100.0), (1e-4, 60.0), (2e-2, 80.0)])
def test_limits_allow_for_the_position_tails(env, sigma, half):
    """Positions up to `half` metres from the grid's centre, where a float coordinate is off by up to 4 um."""
    O, G, ctx, dev = env
    rng = np.random.default_rng(int(half))
    n = 3000
    T = D.rigid(np.linalg.qr(np.random.default_rng(3).normal(size=(3, 3)))[0], np.array([1.0, -2.0, 0.5]))
    if np.linalg.det(T[:3, :3]) < 0:
        T[:3, :3] *= -1.0
    x = rng.uniform(-half, half, (n, 3))
    x = x[np.linalg.norm(x, axis=1) > 3.0].astype(np.float32).astype(np.float64)
    n = len(x)
    k, u = rng.integers(0, 3, n), rng.uniform(0.985, 1.0, n) * rng.choice([-1.0, 1.0], n)
    p = x.copy()
    p[np.arange(n), k] += 3.0 * np.sqrt(2.0) * sigma * u
    iso = lambda m, s: np.tile((s * s * np.eye(3))[SIX], (m, 1)).astype(np.float32)
    tx, tc = np.concatenate([x, np.zeros((1, 3))]), np.concatenate([iso(n, sigma), iso(1, max(0.05, 8 * sigma))])
    case = _case(O, G, ctx, dev, tx, tc, p @ T[:3, :3].T + T[:3, 3], iso(n, sigma))
    r = G.gcvo_eval(ctx, case.grid, *case.src, T)
    o = O.evaluate(case.prob, T, case.kp_o)
    case.grid.close()
    assert o.n_kept > 0.5 * n
    assert abs(r.n_kept - o.n_kept) <= o.n_near_cut, (r.n_kept, o.n_kept, o.n_near_cut)
    assert rel_f_near(r.f, o) < TOL
