"""What the library's host code asks of the CUDA runtime, against a stand-in for
it that runs no kernel (fake_cudart.cpp): the library's objects are linked with
the stand-in and called in a process of their own."""
import glob
import json
import os
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

CHILD = r"""
import ctypes, json, sys
import numpy as np
import torch
sys.path.insert(0, sys.argv[1])
from paper_2606_10019_gb300 import gcvo as G
G.LIB_PATH = sys.argv[2]
L = G.lib()
L.fake_log.restype = ctypes.c_char_p


def log():
    out = [l.split() for l in L.fake_log().decode().splitlines()]
    L.fake_clear()
    return [(int(d), name, int(grid), int(cluster)) for d, name, grid, cluster in out]


def cloud(n):
    return np.random.default_rng(n).normal(size=(3, n)).astype(np.float32)


def problem(ctx, n_src, n_tgt, feat=1, **kw):
    kp = G.kernel_params(eig_max=0.01, feat_dim=feat, cell_size=1.0, **kw)
    cov = lambda n: np.tile(np.float32([1, 0, 0, 1, 0, 1])[:, None], n)
    f = lambda n: np.ones((feat, n), np.float32)
    return G.gcvo_build_grid(ctx, cloud(n_tgt), cov(n_tgt), f(n_tgt), kp), cloud(n_src), cov(n_src), f(n_src), np.eye(4)


"""


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    from paper_2606_10019_gb300 import build as B
    lib = B.build()
    out = str(tmp_path_factory.mktemp("fake") / "libgcvo_fake.so")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(B._nvcc()))), "include")
    objs = glob.glob(os.path.join(os.path.dirname(lib), "*.o"))
    r = subprocess.run(["g++", "-shared", "-fPIC", "-O1", "-Wl,-Bsymbolic", "-I", cuda, "-o", out, os.path.join(HERE, "fake_cudart.cpp")] + objs,
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]

    def run(code):
        r = subprocess.run([sys.executable, "-c", CHILD + code, ROOT, out], capture_output=True, text=True, timeout=300)
        assert r.returncode == 0, r.stderr[-3000:]
        return json.loads(r.stdout.splitlines()[-1])

    return run


def test_every_device_is_set_up(fake):
    """Kernels with more shared memory or larger clusters than the default on the second device used in a process."""
    out = fake(r"""
res = []
for d in (0, 1):
    ctx = G.gcvo_create(d)
    for n in (1500, 5000, 9000, 20000, 40000, 70000):
        G.gcvo_estimate_covariances(ctx, cloud(n), G.kernel_params(eig_max=0.01), np.zeros((6, n), np.float32))
    for feat in (1, 7):
        for n in (1500, 20000):
            p = problem(ctx, n, 1600, feat)
            G.gcvo_eval(ctx, *p)
            G.gcvo_eval_exact(ctx, *p)
            for order in (1, 2, 3):
                G.gcvo_register(ctx, *p, G.solver_params(order=order, k_max=3))
    P = G.Proposal(ctx)
    z, f = torch.zeros((2, 3, 300)), torch.zeros((2, 300))     # (the stand-in's device memory is host memory)
    P.train_step(z, f, z, f, np.tile(np.eye(4), (2, 1, 1)), 1e-3)
    res.append([x[1:] for x in log() if x[0] == d])
print(json.dumps(res))
""")
    assert out[0] == out[1] and len(out[0]) > 100


@pytest.mark.parametrize("most", [1, 2, 8, 16])
def test_clusters_that_cannot_be_placed(fake, most):
    """On a device that places no cluster of more than `most` blocks every size still runs, through clusters of at
    most that size or the grid-wide kernels; with 16 nothing up to 65,536 points leaves the clusters."""
    out = fake(f"most = {most}" + r"""
L.fake_limits(most, 1 << 30)
ctx = G.gcvo_create(0)
for n in (1500, 4000, 9000, 20000, 65536):
    G.gcvo_estimate_covariances(ctx, cloud(n), G.kernel_params(eig_max=0.01), np.zeros((6, n), np.float32))
    p = problem(ctx, n, 1600)
    G.gcvo_eval(ctx, *p)
    G.gcvo_register(ctx, *p, G.solver_params(k_max=3))
    if n <= 20000:
        G.gcvo_register_batched(ctx, [p, p], G.solver_params(k_max=3))
print(json.dumps(log()))
""")
    assert max(x[3] for x in out) == {1: 1, 2: 1, 8: 8, 16: 16}[most]     # 4,000 keys take 4 blocks, 8,000 8, 9,000 16
    assert any("rs_hist" in x[1] for x in out) == any("k_knn_box" in x[1] for x in out) == (most < 16)
    assert any("k_src_keys" in x[1] for x in out) and any("k_src_one" in x[1] for x in out)


def test_cooperative_grid_that_does_not_fit(fake):
    """A register loop whose grid cannot be resident at once replays the graphs."""
    out = fake(r"""
res = []
for coop in (1 << 30, 100):
    L.fake_limits(16, coop)
    ctx = G.gcvo_create(0)
    p = problem(ctx, 20000, 1600)
    log()
    G.gcvo_register(ctx, *p, G.solver_params(k_max=30))
    res.append(log())
print(json.dumps(res))
""")
    loop, graph = (["k_loop" in x[1] for x in r] for r in out)
    assert sum(loop) == 1 and not any(graph)
    assert not any(x[1] == "graph" for x in out[0]) and any(x[1] == "graph" for x in out[1])


@pytest.mark.parametrize("n_src,n_tgt,feat,sub,loop", [(64, 3300000, 7, 32, True), (64, 3400000, 7, 32, False),
                                                       (20, 3400000, 7, 32, True), (3000, 3400000, 7, 8, True),
                                                       (200000, 1200000, 7, 8, False)])
def test_work_items_too_long_for_a_barrier(fake, n_src, n_tgt, feat, sub, loop):
    """The pairs of one warp's last work items bound the register loop's kernel as well as those of the whole set."""
    out = fake(f"n_src, n_tgt, feat, sub = {n_src}, {n_tgt}, {feat}, {sub}" + r"""
ctx = G.gcvo_create(0)
G.gcvo_pair_schedule(ctx, sub)
G.gcvo_register(ctx, *problem(ctx, n_src, n_tgt, feat), G.solver_params(k_max=3))
print(json.dumps(log()))
""")
    assert any("k_loop" in x[1] for x in out) == loop
    assert any(x[1] == "graph" for x in out) != loop


@pytest.mark.parametrize("n_src,pairs,k_max,cutoff,least,most", [(1000, 2, 100, 3.0, 1, 1), (1000, 2, 300, 3.0, 2, 10),
                                                                 (200000, 5, 90, 3.0, 9, 30), (9000, 6, 40, 0.0, 10, 40)])
def test_register_loop_gives_the_gpu_back(fake, n_src, pairs, k_max, cutoff, least, most):
    """The loop's kernel holds every SM, so a launch of it is some milliseconds of iterations, fewer on large sets."""
    out = fake(f"n_src, pairs, k_max, cutoff = {n_src}, {pairs}, {k_max}, {cutoff}" + r"""
ctx = G.gcvo_create(0)
G.gcvo_pair_schedule(ctx, 8)
p = problem(ctx, n_src, 9000, cutoff=cutoff)
G.gcvo_register_batched(ctx, [p] * pairs, G.solver_params(k_max=k_max))
print(json.dumps(log()))
""")
    assert least <= sum("k_loop" in x[1] for x in out) <= most
