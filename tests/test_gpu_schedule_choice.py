"""A call that ends with a non-finite input leaves the choice of the pair pass's
schedule to the first call that does work: that call still times the candidates
(it launches as many kernels as on a fresh context), the next one does not."""
import numpy as np
import pytest

from helpers import soa
from paper_2606_10019_gb300 import datagen as D

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("register", [False, True])
def test_non_finite_input_decides_no_schedule(register):
    import torch
    from paper_2606_10019_gb300 import build as B
    from paper_2606_10019_gb300 import gcvo as G
    B.build()
    dev = torch.device("cuda:0")
    p = D.make_corner_pair(n_src=2500, n_tgt=2400, frame=2)
    kp = G.kernel_params(eig_max=0.01)

    def launches(first_bad):
        ctx = G.gcvo_create(0)
        xyz = [soa(p.tgt_xyz, dev), soa(p.src_xyz, dev)]
        cov = [torch.empty((6, x.shape[1]), device=dev) for x in xyz]
        for x, c in zip(xyz, cov):
            G.gcvo_estimate_covariances(ctx, x, kp, c)
        grid = G.gcvo_build_grid(ctx, xyz[0], cov[0], soa(p.tgt_feat, dev), kp)
        bad = xyz[1].clone()
        bad[2, 77] = float("inf")

        def call(x):
            n0 = G.gcvo_profile_read(ctx)["n_launches"]
            args = (ctx, grid, x, cov[1], soa(p.src_feat, dev), np.eye(4))
            if register:
                G.gcvo_register(*args, G.solver_params(k_max=3, eps_tol=0.0))
            else:
                G.gcvo_eval(*args)
            return G.gcvo_profile_read(ctx)["n_launches"] - n0

        if first_bad:
            with pytest.raises(G.GcvoError) as e:
                call(bad)
            assert e.value.status == G.GCVO_ERR_NONFINITE
        out = call(xyz[1]), call(xyz[1])
        grid.close()
        ctx.close()
        return out

    fresh, after = launches(False), launches(True)
    assert fresh[0] > fresh[1]
    assert after == fresh
