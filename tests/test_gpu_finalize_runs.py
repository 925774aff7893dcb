"""The finalize over many chunks, where a block takes several consecutive ones
and counts those of a problem together: batches of large problems with small
ones of a single chunk between them, in the register loop's kernel and in the
graphs, equal to the same problems registered alone, bit for bit."""
import numpy as np
import pytest

from test_gpu_register_loop import _problem, env  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("profiled", [False, True])
def test_many_chunks_equal_single_problems(env, profiled):
    G, ctx, dev = env
    kinds = [_problem(G, ctx, dev, n, f) for f, n in enumerate((50000, 20, 3000, 40, 17000))]
    order = ([0, 1, 2, 0, 3, 1, 4, 0, 0, 2] * 12)[:-3]
    sp = G.solver_params(k_max=3, eps_tol=1e-12)
    try:
        G.gcvo_pair_schedule(ctx, 4)
        one = [G.gcvo_register(ctx, *p, sp) for p in kinds]
        G.gcvo_profile_enable(ctx, profiled)
        T, logs, n_iter, status = G.gcvo_register_batched(ctx, [kinds[k] for k in order], sp, want_log=True)
    finally:
        G.gcvo_profile_enable(ctx, False)
        G.gcvo_pair_schedule(ctx, 0)
    for k, Tk, lg, n, st in zip(order, T, logs, n_iter, status):
        assert np.array_equal(Tk, one[k][0]) and n == one[k][2] and st == one[k][3]
        assert lg.tobytes() == one[k][1].tobytes()
