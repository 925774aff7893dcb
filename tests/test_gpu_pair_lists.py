"""The pair pass's two target lists -- pairs counted whole or one by one, pairs
evaluated within the per-axis and norm bounds -- against the FP64 oracle:
flat and round covariances an order below the problem's largest, tilted
planes, clouds at the grid's centre and far from it, single points and full
sub-tiles.  Tolerances: the repository's 1e-5 on f and g less the terms of the
pairs within rounding of the cutoff; counts equal up to the pairs within
float32 rounding of rho and of the cutoff."""
from types import SimpleNamespace

import numpy as np
import pytest

from helpers import Case, rel_f_near, rel_g_near
from paper_2606_10019_gb300 import datagen as D
from test_gpu_parity import TOL, _rho_count_bounds, env  # noqa: F401

pytestmark = pytest.mark.gpu


def _covs(rng, normals, flat, thick):
    """Sigma = thick^2 I + (flat^2 - thick^2) (I - n n^T), six per point."""
    P = np.eye(3)[None] - normals[:, :, None] * normals[:, None, :]
    C = thick ** 2 * np.eye(3)[None] + (flat ** 2 - thick ** 2) * P
    return C[:, [0, 0, 0, 1, 1, 2], [0, 1, 2, 1, 2, 2]].astype(np.float32)


@pytest.mark.parametrize("n,flat,thick,offset,tilt", [
    (1, 0.05, 0.005, 0.0, 0.0), (33, 0.05, 0.05, 0.0, 0.3), (900, 0.04, 0.004, 0.0, 0.0),
    (900, 0.04, 0.004, 0.0, 0.5), (900, 0.03, 0.03, 0.0, 0.2), (900, 0.04, 0.01, 60.0, 0.5),
    (900, 0.02, 0.002, 60.0, 0.0)])
def test_lists_match_oracle(env, n, flat, thick, offset, tilt):
    O, G, ctx, dev = env
    rng = np.random.default_rng(n + int(1e4 * flat) + int(10 * tilt))
    R = np.linalg.qr(np.eye(3) + tilt * rng.normal(size=(3, 3)))[0]

    def cloud(m):
        k = rng.integers(0, 3, m)
        x = rng.uniform(0, 1.0, (m, 3))
        x[np.arange(m), k] = thick * rng.normal(size=m)
        return x @ R.T + offset * np.array([1.0, 0.6, 0.1]), np.eye(3)[k] @ R.T

    tx, tn = cloud(2500)
    sx, sn = cloud(n)
    tc, sc = _covs(rng, tn, flat, thick), _covs(rng, sn, flat, thick)
    # one far target with a covariance 25 times as large sets rho for all
    far = np.array([[1.0, 0.6, 0.1]]) * offset + (np.full((1, 3), 30.0) if offset else np.full((1, 3), 3.0))
    tx, tc = np.concatenate([tx, far]), np.concatenate([tc, 25 * _covs(rng, np.eye(3)[:1], flat, flat)])
    pair = SimpleNamespace(tgt_xyz=tx.astype(np.float32), src_xyz=sx.astype(np.float32),
                           tgt_feat=rng.uniform(0.5, 1, (len(tx), 1)).astype(np.float32),
                           src_feat=rng.uniform(0.5, 1, (n, 1)).astype(np.float32))
    case = Case(O, pair, O.KernelParams(cutoff=3.0), iso=True)
    case.iso, case.tc, case.sc = False, tc, sc
    case.prob = O.Problem.make(pair.tgt_xyz, tc, pair.tgt_feat, pair.src_xyz, sc, pair.src_feat)
    case.gpu(G, ctx, dev, G.kernel_params(eig_max=0.01))
    T = D.rigid(np.eye(3), np.array([0.01, -0.006, 0.008]))
    o = O.evaluate(case.prob, T, case.kp_o)
    out = []
    try:
        for sub in (4, 8, 16, 32):
            G.gcvo_pair_schedule(ctx, sub)
            out.append(G.gcvo_eval(ctx, case.grid, *case.src, T))
    finally:
        G.gcvo_pair_schedule(ctx, 0)
    case.grid.close()
    assert len({(int(r.n_pairs), int(r.n_kept)) for r in out}) == 1
    lo, hi = _rho_count_bounds(O, case, T, out[0].rho)
    assert lo <= out[0].n_pairs <= hi
    assert abs(out[0].n_kept - o.n_kept) <= o.n_near_cut
    for r in out:
        assert rel_f_near(r.f, o) < TOL and rel_g_near(r.g, o) < TOL
