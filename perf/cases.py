"""The work that users of this library have it do, as cases that can be timed and checked.

A case goes through the public entry points of `paper_2606_10019_gb300.gcvo`, as a program that
tracks frames, refines batches of poses or trains the initial-pose proposal calls them.  Sizes
and options are those of the repository's benchmark and tests: corner scenes of 400 to 40,000
points, 64-beam LiDAR frames in 0.3 m voxels, RGB-D frames in 2 cm voxels, batches of up to 64
uneven problems, and 256 pairs of 4096 points for the proposal.

One context per process serves every state, as in a program that keeps it from frame to frame.
The point covariances that an evaluation is given are made here in 64 bits and rounded to
float32, so that they do not depend on the library.  The library sums float32 pair terms (and
float32 / bfloat16 network products): outputs of that accuracy are returned in float32, although
the C ABI hands some of them out in double variables; counts are returned as whole numbers.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2606_10019_gb300 import datagen as D
from paper_2606_10019_gb300 import gcvo as G
from paper_2606_10019_gb300 import train_proposal as TP

DEV = "cuda:0"
KNN, EIG_RATIO, CUTOFF = 10, 100.0, 3.0
EIG_MAX = {"corner": 0.01, "lidar": 0.09, "rgbd": 4e-4}
ISO_ELL = {"corner": 0.08, "lidar": 0.2, "rgbd": 0.02}
MOST = {"corner": 40000, "lidar": 20000, "rgbd": 20000}     # points of a cloud
# how far from the truth a pose is in the middle of a registration: degrees, metres
OFF = {"corner": (2.0, 0.05), "lidar": (0.3, 0.1), "rgbd": (0.3, 0.01)}
# pairs that pass the cutoff, per source point, at these poses and MOST target points (measured);
# a thinner cloud has wider covariances, so the number falls slowly with its size
KEPT, THIN = {"corner": 23.0, "lidar": 18.0, "rgbd": 30.0}, 0.2

_ctx = None


def context():
    global _ctx
    if _ctx is None:
        _ctx = G.gcvo_create(0)
    return _ctx


def listed():
    return [
        # the smallest call: one evaluation of a few hundred points, all latency
        {"name": "eval corner 400", "kind": "eval", "scene": "corner", "n_src": 400, "n_tgt": 371, "feat": 1,
         "iso": False, "dense": False},
        # one evaluation of a LiDAR frame against the previous one
        {"name": "eval lidar frame", "kind": "eval", "scene": "lidar", "n_src": 19997, "n_tgt": 20000, "feat": 1,
         "iso": False, "dense": False},
        # one evaluation of an RGB-D frame with its colours
        {"name": "eval rgbd frame", "kind": "eval", "scene": "rgbd", "n_src": 19999, "n_tgt": 19501, "feat": 3,
         "iso": False, "dense": False},
        # the densest pair of clouds of the uneven batch
        {"name": "eval corner 40k", "kind": "eval", "scene": "corner", "n_src": 40000, "n_tgt": 39001, "feat": 1,
         "iso": False, "dense": False},
        # the exact Riemannian Hessian (G-CVO-E) of a LiDAR frame pair
        {"name": "exact lidar frame", "kind": "exact", "scene": "lidar", "n_src": 19997, "n_tgt": 20000, "feat": 1,
         "iso": False, "dense": False},
        # covariances of one frame, as a tracker takes them of every new frame
        {"name": "covariances lidar frame", "kind": "cov", "scene": "lidar", "clouds": 1, "n_min": 19999,
         "n_max": 19999, "knn": 10},
        # covariances of the clouds of a batch: sizes of 1,000 to 40,000, corner scenes and frames in turn
        {"name": "covariances 32 clouds", "kind": "cov", "scene": "mixed", "clouds": 32, "n_min": 1000,
         "n_max": 40000, "knn": 10},
        # the plain example: two clouds of 2000 points registered from the identity, grid at hand
        {"name": "register corner 2000", "kind": "register", "scene": "corner", "n_src": 2000, "n_tgt": 2000,
         "feat": 1, "iso": False},
        # frame-to-frame tracking: raw clouds in, pose out, from a motion model's prediction
        {"name": "track lidar frame", "kind": "clouds", "scene": "lidar", "pairs": 1, "n_min": 20000,
         "n_max": 20000},
        # batched refinement of problems of uneven size, raw clouds in, poses out
        {"name": "refine 64 pairs", "kind": "clouds", "scene": "mixed", "pairs": 64, "n_min": 1000, "n_max": 40000},
        # the proposal network: poses for a batch of pairs, and one training step on a batch
        {"name": "propose 256 x 4096", "kind": "propose", "pairs": 256, "n": 4096},
        {"name": "train 256 x 4096", "kind": "train", "pairs": 256, "n": 4096},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["eval", "eval", "exact", "cov", "register", "clouds", "propose", "train"])
    scene = rng.choice(["corner", "lidar", "rgbd"])
    if kind in ("eval", "exact", "register"):
        most = MOST[scene] if kind == "eval" else 20000
        least = 371 if scene == "corner" else 1000
        if kind == "register" and scene == "rgbd":
            scene = "corner"
        n = _log_int(rng, least, most)
        c = {"kind": kind, "scene": scene, "n_src": n, "n_tgt": min(most, max(least, int(n * rng.uniform(0.8, 1.25)))),
             "feat": 3 if scene == "rgbd" else rng.choice([1, 1, 1, 3, 5]), "iso": rng.random() < 0.2}
        if kind == "register":
            c["feat"] = 1
        else:
            c["dense"] = rng.random() < 0.15 and n <= 5000
        return c
    if kind == "cov":
        lo = _log_int(rng, 1000, 20000)
        one = rng.random() < 0.5
        return {"kind": "cov", "scene": scene if one else "mixed", "clouds": 1 if one else _log_int(rng, 2, 32),
                "n_min": lo, "n_max": lo if one else 2 * lo, "knn": rng.choice([6, 10, 10, 10, 13, 16])}
    if kind == "clouds":
        lo = _log_int(rng, 1000, 20000)
        one = rng.random() < 0.4
        return {"kind": "clouds", "scene": rng.choice(["corner", "lidar"]) if one else "mixed",
                "pairs": 1 if one else _log_int(rng, 2, 48), "n_min": lo, "n_max": lo if one else 2 * lo}
    return {"kind": kind, "pairs": _log_int(rng, 1, 256), "n": _log_int(rng, 200, 4096)}


# --------------------------------------------------------------------------------------------
# Scenes, made on the GPU in 64 bits from the generators' streets and rooms.
# --------------------------------------------------------------------------------------------

def _t(a):
    return torch.as_tensor(np.asarray(a, dtype=np.float64), device=DEV)


def _first_box(o, d, lo, hi):
    """Distance along d to the first box that each ray from o enters (inf: none), which, and its face's axis."""
    inv = 1.0 / torch.where(d.abs() > 1e-12, d, torch.full_like(d, 1e-12))
    best = torch.full((len(d),), math.inf, dtype=torch.float64, device=DEV)
    which = torch.zeros(len(d), dtype=torch.int64, device=DEV)
    axis = torch.zeros_like(which)
    for k in range(0, len(lo), 32):
        a = (lo[k:k + 32, None] - o) * inv
        b = (hi[k:k + 32, None] - o) * inv
        near, ax = torch.minimum(a, b).max(-1)
        far = torch.maximum(a, b).min(-1).values
        near = torch.where((near <= far) & (near > 1e-6), near, math.inf)
        m, w = near.min(0)
        up = m < best
        best = torch.where(up, m, best)
        which = torch.where(up, w + k, which)
        axis = torch.where(up, ax.gather(0, w[None])[0], axis)
    return best, which, axis


def _voxels(xyz, feat, edge):
    """Centroid and mean feature of every occupied voxel."""
    key = torch.floor(xyz / edge).long()
    key -= key.min(0).values
    dims = key.max(0).values + 1
    lin = (key[:, 0] * dims[1] + key[:, 1]) * dims[2] + key[:, 2]
    _, inv, cnt = torch.unique(lin, return_inverse=True, return_counts=True)
    both = torch.cat([xyz, feat], 1)
    out = torch.zeros((len(cnt), both.shape[1]), dtype=torch.float64, device=DEV).index_add_(0, inv, both)
    out = (out / cnt[:, None]).float()
    return out[:, :3], out[:, 3:]


def _lidar_frame(street, pose, gen):
    """One 64 x 1800 scan of a street (ground, boxes, poles, porous crowns), 0.3 m voxels."""
    el, az = torch.meshgrid(_t(D.LIDAR_ELEV), _t(D.LIDAR_AZ), indexing="ij")
    ds = torch.stack([el.cos() * az.cos(), el.cos() * az.sin(), el.sin()], -1).reshape(-1, 3)
    o, d = _t(pose[:3, 3]), ds @ _t(pose[:3, :3]).T
    near = np.abs(street.poles[:, 0] - pose[0, 3]) < D.LIDAR_RANGE
    pl = street.poles[near]
    r = street.pole_r
    box = (street.boxes_lo[:, 0] < pose[0, 3] + D.LIDAR_RANGE) & (street.boxes_hi[:, 0] > pose[0, 3] - D.LIDAR_RANGE)
    lo = np.concatenate([street.boxes_lo[box], np.c_[pl - r, np.zeros(len(pl))]])
    hi = np.concatenate([street.boxes_hi[box], np.c_[pl + r, np.full(len(pl), street.pole_h)]])
    inten = _t(np.concatenate([street.box_int[box], np.full(len(pl), 0.9)]))
    t, which, axis = _first_box(o, d, _t(lo), _t(hi))
    base, cosine = inten[which], d.gather(1, axis[:, None])[:, 0].abs()
    g = torch.where(d[:, 2] < -1e-9, -o[2] / d[:, 2], math.inf)
    base, cosine = torch.where(g < t, 0.3, base), torch.where(g < t, d[:, 2].abs(), cosine)
    t = torch.minimum(t, g)
    c = _t(street.crowns[np.abs(street.crowns[:, 0] - pose[0, 3]) < D.LIDAR_RANGE + 5.0])
    for k in range(0, len(c), 32):
        oc = o - c[k:k + 32, :3]
        b = oc @ d.T
        disc = b * b - ((oc * oc).sum(1) - c[k:k + 32, 3] ** 2)[:, None]
        sq = disc.clamp(min=0).sqrt()
        depth = torch.empty_like(b).exponential_(1.0 / 0.7, generator=gen)
        hit = (-b - sq).clamp(min=1e-6) + depth
        hit = torch.where((disc > 0) & (hit < -b + sq), hit, math.inf).min(0).values
        base, cosine = torch.where(hit < t, 0.15, base), torch.where(hit < t, 0.5, cosine)
        t = torch.minimum(t, hit)
    ok = t <= D.LIDAR_RANGE
    t = t[ok] + 0.01 * torch.randn(int(ok.sum()), generator=gen, device=DEV, dtype=torch.float64)
    pts = ds[ok] * t[:, None]
    f = (0.75 * base + 0.25 * cosine)[ok, None]
    n_out = len(pts) // 100
    u = torch.rand((n_out, 4), generator=gen, device=DEV, dtype=torch.float64)
    out = pts.min(0).values + u[:, :3] * (pts.max(0).values - pts.min(0).values)
    return _voxels(torch.cat([pts, out]), torch.cat([f, u[:, 3:]]), 0.3)


def _rgbd_frame(room, pose, gen):
    """One 640 x 480 depth and colour frame of a room, 2 cm voxels."""
    v, u = torch.meshgrid(_t(np.arange(480)), _t(np.arange(640)), indexing="ij")
    dc = torch.stack([(u - 319.5) / 525.0, (v - 239.5) / 525.0, torch.ones_like(u)], -1).reshape(-1, 3)
    z, which, _ = _first_box(_t(pose[:3, 3]), dc @ _t(pose[:3, :3]).T, _t(room.lo), _t(room.hi))
    ok = z < 8.0
    z = z[ok]
    z = z + torch.randn(len(z), generator=gen, device=DEV, dtype=torch.float64) * 0.0012 * z * z
    return _voxels(dc[ok] * z[:, None], _t(room.rgb)[which[ok]], 0.02)


def _take(xyz, feat, n, gen):
    if len(xyz) > n:
        at = torch.randperm(len(xyz), generator=gen, device=DEV)[:n].sort().values
        xyz, feat = xyz[at], feat[at]
    return xyz.contiguous(), feat.contiguous()


def _frames(scene, seed, gen):
    """Two consecutive frames of a sequence of its own street or room, and their motion (T^-1 z ~ x)."""
    seq = (D.LidarSequence if scene == "lidar" else D.RgbdSequence)(n_frames=2, stream=10 + seed)
    a, b = seq.poses
    frame = (lambda p: _lidar_frame(seq.street, p, gen)) if scene == "lidar" else (lambda p: _rgbd_frame(seq.room, p, gen))
    return frame(a), frame(b), D.inv_rigid(b) @ a


def _pair(scene, n_src, n_tgt, seed, gen, frames=None):
    """(target xyz, target feat, source xyz, source feat, T_true): (n, 3) and (n, l) float32 on the GPU."""
    if scene == "corner":
        p = D.make_corner_pair(frame=seed, n_src=n_src, n_tgt=n_tgt, stream=10)
        g = lambda a: torch.from_numpy(a).to(DEV)
        return g(p.tgt_xyz), g(p.tgt_feat), g(p.src_xyz), g(p.src_feat), p.T_true
    (tx, tf), (sx, sf), T = frames or _frames(scene, seed, gen)
    return (*_take(tx, tf, n_tgt, gen), *_take(sx, sf, n_src, gen), T)


def _perturbed(T, scene, seed, times=1.0):
    deg, met = OFF[scene]
    rng = np.random.default_rng([seed, 77])
    return D.random_motion(rng, times * deg, times * met) @ T


def _covariances(xyz, knn, eig_max):
    """Eq. (7b) and the eigenvalue bound of n points (n, 3), in 64 bits: (n, 6)."""
    x = xyz.double()
    out = []
    step = max(1, (1 << 26) // len(x))
    for k in range(0, len(x), step):
        q = x[k:k + step]
        d2 = sum((q[:, a, None] - x[None, :, a]) ** 2 for a in range(3))
        y = x[d2.topk(knn, largest=False).indices] - q[:, None]
        out.append(torch.einsum("nka,nkb->nab", y, y) / (knn - 1))
    S = torch.cat(out)
    # eigenvectors on the host: a batched 3 x 3 solver in 64 bits
    w, V = np.linalg.eigh(S.cpu().numpy())
    w = np.clip(w, eig_max / EIG_RATIO, eig_max)
    B = np.einsum("nak,nk,nbk->nab", V, w, V)
    return _t(B.reshape(-1, 9)[:, [0, 1, 2, 4, 5, 8]])


def _soa(a):
    return a.float().T.contiguous()


def _params(case, scene, **kw):
    return G.kernel_params(kernel_mode=1 if case.get("iso") else 0, cutoff=0.0 if case.get("dense") else CUTOFF,
                           iso_ell=ISO_ELL[scene], knn=case.get("knn", KNN), eig_max=EIG_MAX[scene],
                           eig_ratio=EIG_RATIO, feat_dim=case.get("feat", 1), **kw)


def _features(f, feat, gen):
    """feat channels: the scene's own, or a label distribution over `feat` classes."""
    if f.shape[1] == feat:
        return f
    p = torch.rand((len(f), feat), generator=gen, device=DEV).pow(3) + 1e-3
    return p / p.sum(1, keepdim=True)


def _generator(seed):
    return torch.Generator(device=DEV).manual_seed(seed)


def _single(case, seed):
    """The two clouds of an evaluation or a registration, with covariances, and a pose."""
    gen = _generator(seed)
    scene = case["scene"]
    tx, tf, sx, sf, T = _pair(scene, case["n_src"], case["n_tgt"], seed, gen)
    tf, sf = _features(tf, case["feat"], gen), _features(sf, case["feat"], gen)
    tc = sc = None
    if not case["iso"]:
        tc, sc = (_covariances(x, KNN, EIG_MAX[scene]).float() for x in (tx, sx))
    if case["kind"] == "register":
        T0 = np.eye(4) if scene == "corner" else _perturbed(T, scene, seed)
    else:
        T0 = _perturbed(T, scene, seed)
    return tx, tc, tf, sx, sc, sf, T0


def _kinds(case, count, seed):
    """Scene and size of each cloud (or pair) of a batch: sizes spread evenly over the logarithm of the range."""
    order = np.random.default_rng([len(case), count]).permutation(count)
    for k in range(count):
        at = (order[k] + 0.5) / count
        n = int(round(math.exp(math.log(case["n_min"]) * (1 - at) + math.log(case["n_max"]) * at)))
        scene = case["scene"] if case["scene"] != "mixed" else ("corner", "lidar")[k % 2]
        yield k, scene, min(n, MOST[scene])


def _clouds(case, seed):
    gen = _generator(seed)
    frames = {}
    for k, scene, n in _kinds(case, case["clouds"], seed):
        if scene != "corner" and scene not in frames:
            frames[scene] = _frames(scene, seed, gen)
        yield _pair(scene, 16, n, seed + 7919 * k, gen, frames.get(scene))[0], scene


def _cloud_pairs(case, seed):
    gen = _generator(seed)
    frames = None
    for k, scene, n in _kinds(case, case["pairs"], seed):
        if scene != "corner" and frames is None:
            frames = _frames(scene, seed, gen)
        tx, tf, sx, sf, T = _pair(scene, n, n, seed + 7919 * k, gen, frames)
        yield scene, tx, tf, sx, sf, _perturbed(T, scene, seed + 7919 * k)


def _proposal_batch(case, seed):
    """Pairs of corner scenes misaligned by up to 30 degrees and half a metre, and their poses."""
    gen = _generator(seed)
    B, n = case["pairs"], case["n"]
    rng = np.random.default_rng([seed, 3])
    rand = lambda *s: torch.rand(s, generator=gen, device=DEV, dtype=torch.float64)
    randn = lambda *s: torch.randn(s, generator=gen, device=DEV, dtype=torch.float64)

    def scene():
        which = torch.multinomial(_t([4.0, 4.0, 4.0, math.pi]), B * n, replacement=True, generator=gen)
        uv = 2.0 * rand(B * n, 3)
        ball = randn(B * n, 3)
        ball = 1.0 + 0.5 * ball / ball.norm(dim=1, keepdim=True)
        flat = uv * (torch.arange(3, device=DEV) != which[:, None])
        return torch.where((which == 3)[:, None], ball, flat).reshape(B, n, 3)

    T = np.stack([D.perturb(rng, 30.0, 0.5) for _ in range(B)])
    R, t = _t(T[:, :3, :3]), _t(T[:, :3, 3])
    tgt = scene() + 0.01 * randn(B, n, 3)
    src = torch.einsum("bij,bnj->bni", R, scene()) + t[:, None] + 0.01 * randn(B, n, 3)
    soa = lambda a: a.transpose(1, 2).float().contiguous()
    return soa(src), rand(B, n).float(), soa(tgt), rand(B, n).float(), T


def _weights(seed):
    return TP.init_params(int(sum(r * c for r, c in NET)), seed)


# --------------------------------------------------------------------------------------------
# prepare, run
# --------------------------------------------------------------------------------------------

def prepare(case, seed):
    ctx, kind = context(), case["kind"]
    s = {"kind": kind, "ctx": ctx}
    if kind in ("eval", "exact", "register"):
        tx, tc, tf, sx, sc, sf, T0 = _single(case, seed)
        c = lambda a: None if a is None else _soa(a)
        s["grid"] = G.gcvo_build_grid(ctx, _soa(tx), c(tc), _soa(tf), _params(case, case["scene"]))
        s["src"] = (_soa(sx), c(sc), _soa(sf))
        s["T"] = T0
        s["solver"] = G.solver_params(k_max=200, eps_tol=1e-6)
    elif kind == "cov":
        clouds = list(_clouds(case, seed))
        s["xyz"] = [_soa(x) for x, _ in clouds]
        s["cov"] = [torch.empty((6, len(x)), device=DEV) for x, _ in clouds]
        # one eigenvalue bound for a batched call, as its parameters are the call's
        s["kp"] = _params({"knn": case["knn"]}, "lidar" if case["scene"] == "mixed" else case["scene"])
    elif kind == "clouds":
        s["pairs"] = [(_soa(tx), _soa(tf), _soa(sx), _soa(sf), T0, _params({}, scene))
                      for scene, tx, tf, sx, sf, T0 in _cloud_pairs(case, seed)]
        s["kp"] = s["pairs"][0][5]
        s["solver"] = G.solver_params(k_max=200, eps_tol=1e-6)
    else:
        s["net"] = G.Proposal(ctx)
        s["net"].set_params(_weights(seed % 1000))
        *s["batch"], s["T"] = _proposal_batch(case, seed)
    return s


def _f32(a):
    return np.asarray(a, dtype=np.float32)


def run(s):
    kind, ctx = s["kind"], s["ctx"]
    if kind == "eval":
        r = G.gcvo_eval(ctx, s["grid"], *s["src"], s["T"])
        return {"f": _f32(r.f), "g": _f32(r.g), "H": _f32(r.H), "M": _f32(r.M), "n_pairs": r.n_pairs, "n_kept": r.n_kept}
    if kind == "exact":
        r = G.gcvo_eval_exact(ctx, s["grid"], *s["src"], s["T"])
        return {"f": _f32(r.f), "g": _f32(r.g), "H": _f32(r.H), "D": _f32(r.D), "n_pairs": r.n_pairs, "n_kept": r.n_kept}
    if kind == "register":
        T, _, _, _ = G.gcvo_register(ctx, s["grid"], *s["src"], s["T"], s["solver"], want_log=False)
        return {"T": _f32(T)}
    if kind == "cov":
        if len(s["xyz"]) == 1:
            G.gcvo_estimate_covariances(ctx, s["xyz"][0], s["kp"], s["cov"][0])
        else:
            G.gcvo_estimate_covariances_batched(ctx, s["xyz"], s["kp"], s["cov"])
        return s["cov"]
    if kind == "clouds":
        T, _, _, _ = G.gcvo_register_clouds(ctx, s["pairs"], s["kp"], s["solver"])
        return {"T": _f32(T)}
    if kind == "propose":
        twist, T0 = s["net"].infer(*s["batch"])
        return {"twist": twist, "T0": _f32(T0)}
    loss, grad = s["net"].train_step(*s["batch"], s["T"], lr=1e-4, want_grad=True)
    return {"loss": _f32(loss), "grad": grad}


# --------------------------------------------------------------------------------------------
# What a pass cannot do without
# --------------------------------------------------------------------------------------------

NET = [(64, 4), (64, 1), (128, 64), (128, 1), (256, 128), (256, 1), (256, 512), (256, 1), (128, 256), (128, 1),
       (6, 128), (6, 1)]
POINT_FLOPS = 2 * (4 * 64 + 64 * 128 + 128 * 256)
HEAD_FLOPS = 2 * (512 * 256 + 256 * 128 + 128 * 6)
PAIR_FLOPS, EXACT_FLOPS = 76, 232      # float32 operations of one pair that counts
ITERATIONS = 20                        # of a registration, about


def _kept(scene, ns, nt):
    return ns * KEPT[scene] * (nt / MOST[scene]) ** THIN


def work(case):
    kind = case["kind"]
    if kind in ("eval", "exact", "register"):
        ns, nt, fd = case["n_src"], case["n_tgt"], case["feat"]
        pairs = ns * nt if case.get("dense") else _kept(case["scene"], ns, nt)
        times = ITERATIONS if kind == "register" else 1
        # the source's position, covariance and features; the grid's point records
        return {"bytes": 4 * ns * (9 + fd) + 4 * nt * (9 + fd),
                "flops": times * pairs * (EXACT_FLOPS if kind == "exact" else PAIR_FLOPS)}
    if kind == "cov":
        n = sum(m for _, _, m in _kinds(case, case["clouds"], 0))
        # 12 bytes in, 24 out; at least the neighbours' distances and one 3 x 3 eigenproblem
        return {"bytes": 36 * n, "flops": n * (case["knn"] * 20 + 300)}
    if kind == "clouds":
        sizes = [(scene, m) for _, scene, m in _kinds(case, case["pairs"], 0)]
        n = sum(m for _, m in sizes)
        pairs = sum(_kept(scene, m, m) for scene, m in sizes)
        return {"bytes": 2 * 16 * n + 128 * len(sizes), "flops": 2 * n * (KNN * 20 + 300) + ITERATIONS * pairs * PAIR_FLOPS}
    B, n = case["pairs"], case["n"]
    params = sum(r * c for r, c in NET)
    fwd = 2 * B * n * POINT_FLOPS + B * HEAD_FLOPS
    if kind == "propose":
        return {"bytes": 2 * B * n * 16 + 2 * params + B * 152, "flops": fwd}
    # backward: each channel's largest point only
    return {"bytes": 2 * B * n * 16 + 4 * 8 * params, "flops": fwd + 2 * B * 256 * 2 * POINT_FLOPS / 3 + 2 * B * HEAD_FLOPS}


# --------------------------------------------------------------------------------------------
# The same values in 64 bits, from the formulas
# --------------------------------------------------------------------------------------------

def _hat(w):
    z = torch.zeros_like(w[0])
    return torch.stack([torch.stack([z, -w[2], w[1]]), torch.stack([w[2], z, -w[0]]), torch.stack([-w[1], w[0], z])])


def _sym(c):
    return torch.stack([c[:, 0], c[:, 1], c[:, 2], c[:, 1], c[:, 3], c[:, 4], c[:, 2], c[:, 4], c[:, 5]], 1).reshape(-1, 3, 3)


def _gamma(g):
    Gam = torch.zeros((6, 6), dtype=torch.float64, device=DEV)
    Gam[:3, :3], Gam[3:, :3] = -0.5 * _hat(g[:3]), -_hat(g[3:])
    return Gam


class _Dense:
    """f, g, M and D(g) of two clouds over all pairs, chunk by chunk of the source."""

    def __init__(self, tx, tc, tf, sx, sc, sf, iso_ell, cutoff):
        self.t = (tx.double(), None if tc is None else _sym(tc.double()), tf.double())
        self.s = (sx.double(), None if sc is None else _sym(sc.double()), sf.double())
        self.ell, self.cut = iso_ell, cutoff
        top = lambda c: float(np.linalg.eigvalsh(c.cpu().numpy()).max())
        lam = iso_ell ** 2 if tc is None else top(self.t[1]) + top(self.s[1])
        self.reach = math.inf if not cutoff else cutoff ** 2 * lam * (1 + 1e-6)

    def _terms(self, xi, T, z, cz, lz, x, cx, lx):
        """Per pair: weight, lever arm, Sigma^-1 r and Sigma^-1 at T (I + xi^)."""
        R, t = T[:3, :3], T[:3, 3]
        W = torch.eye(3, dtype=torch.float64, device=DEV) - _hat(xi[:3])
        p = (z - t - R @ xi[3:]) @ R @ W.T
        if cz is None:
            A = torch.eye(3, dtype=torch.float64, device=DEV).expand(len(z), 3, 3) / self.ell ** 2
        else:
            Q = R @ W.T
            S = cx + Q.T @ cz @ Q
            c = torch.stack([torch.linalg.cross(S[:, 1], S[:, 2]), torch.linalg.cross(S[:, 2], S[:, 0]),
                             torch.linalg.cross(S[:, 0], S[:, 1])], 1)
            A = c / (S[:, 0] * c[:, 0]).sum(1)[:, None, None]
        r = x - p
        u = torch.einsum("nab,nb->na", A, r)
        d2 = (r * u).sum(1)
        keep = d2.detach() <= self.cut ** 2 if self.cut else torch.ones_like(d2, dtype=torch.bool)
        return (lx * lz).sum(1) * torch.exp(-0.5 * d2) * keep, p, u, A

    def _chunks(self, T):
        R, t = T[:3, :3], T[:3, 3]
        x, cx, lx = self.t
        z, cz, lz = self.s
        p = (z - t) @ R
        step = max(1, (1 << (25 if self.cut else 21)) // len(x))
        for k in range(0, len(z), step):
            q = p[k:k + step]
            j, i = (sum((x[None, :, a] - q[:, a, None]) ** 2 for a in range(3)) <= self.reach).nonzero(as_tuple=True)
            for m in range(0, len(j), 1 << 21):
                a, b = j[m:m + (1 << 21)] + k, i[m:m + (1 << 21)]
                yield z[a], None if cz is None else cz[a], lz[a], x[b], None if cx is None else cx[b], lx[b]

    def eval(self, T, derivative=False):
        T = _t(T)
        xi = torch.zeros(6, dtype=torch.float64, device=DEV)
        f, g = torch.zeros((), dtype=torch.float64, device=DEV), torch.zeros(6, dtype=torch.float64, device=DEV)
        M, Dg = torch.zeros((6, 6), dtype=torch.float64, device=DEV), torch.zeros((6, 6), dtype=torch.float64, device=DEV)

        def grad(xi, *pair):
            w, p, u, _ = self._terms(xi, T, *pair)
            return -(w[:, None] * torch.cat([torch.linalg.cross(p, u), u], 1)).sum(0)

        for pair in self._chunks(T):
            w, p, u, A = self._terms(xi, T, *pair)
            f += w.sum()
            g -= (w[:, None] * torch.cat([torch.linalg.cross(p, u), u], 1)).sum(0)
            J = torch.cat([-_hat(p.T).permute(2, 0, 1), torch.eye(3, dtype=torch.float64, device=DEV).expand(len(p), 3, 3)], 2)
            M += torch.einsum("n,nar,nab,nbs->rs", w, J, A, J) if len(p) < 1 << 16 else ((w[:, None, None] * (A @ J)).transpose(1, 2) @ J).sum(0)
            if derivative:
                Dg += torch.autograd.functional.jacobian(lambda v: grad(v, *pair), xi)
        return f, g, M, Dg

    def register(self, T0, k_max, eps):
        T = np.array(T0, dtype=np.float64)
        for _ in range(k_max):
            _, g, M, _ = self.eval(T)
            xi = torch.linalg.solve(M - _gamma(g), g)
            X = torch.zeros((4, 4), dtype=torch.float64, device=DEV)
            X[:3, :3], X[:3, 3] = _hat(xi[:3]), xi[3:]
            T = T @ torch.matrix_exp(X).cpu().numpy()
            if float(xi.abs().sum()) < eps:
                break
        return T


def _net64(case, seed):
    """The network with bfloat16 weights and layer inputs, sums in 64 bits: the pooled points and what follows."""
    sx, sl, tx, tl, T = _proposal_batch(case, seed)
    w = torch.from_numpy(_weights(seed % 1000)).to(DEV)
    P, at = [], 0
    for r, c in NET:
        P.append(w[at:at + r * c].reshape(r, c))
        at += r * c
    P = [p.bfloat16().double() if k % 2 == 0 else p.double()[:, 0] for k, p in enumerate(P)]
    for p in P:
        p.requires_grad_(True)
    B = case["pairs"]
    x, z = tx.double(), sx.double()
    c = x.mean(2, keepdim=True)
    s = ((x - c) ** 2).sum(1).mean(1).sqrt()[:, None, None] + 1e-6
    pts = torch.stack([torch.cat([(z - c) / s, sl.double()[:, None]], 1), torch.cat([(x - c) / s, tl.double()[:, None]], 1)], 1)
    pts = pts.reshape(2 * B, 4, -1).transpose(1, 2)
    half = lambda a: a + (a.detach().bfloat16().double() - a.detach())

    def points(q):
        h = half(torch.relu(q @ P[0].T + P[1]))
        h = half(torch.relu(h @ P[2].T + P[3]))
        return h

    with torch.no_grad():
        arg = torch.stack([(points(q) @ P[4].T + P[5]).argmax(0) for q in pts])
    top = torch.gather(pts, 1, arg[:, :, None].expand(-1, -1, 4))
    h = points(top)
    feat = (h * P[4]).sum(2) + P[5]
    y = torch.relu(feat.reshape(B, 512) @ P[6].T + P[7])
    y = torch.relu(y @ P[8].T + P[9])
    return y @ P[10].T + P[11], P, T, c[:, :, 0].detach().cpu().numpy(), s[:, 0, 0].detach().cpu().numpy()


def _exp_se3(xi):
    X = np.zeros((4, 4))
    X[:3, :3] = [[0, -xi[2], xi[1]], [xi[2], 0, -xi[0]], [-xi[1], xi[0], 0]]
    X[:3, 3] = xi[3:]
    return torch.matrix_exp(torch.from_numpy(X)).numpy()


def _log_se3(T):
    from scipy.spatial.transform import Rotation
    w = Rotation.from_matrix(T[:3, :3]).as_rotvec()
    W = np.array([[0, -w[2], w[1]], [w[2], 0, -w[0]], [-w[1], w[0], 0]])
    th = np.linalg.norm(w)
    V = np.eye(3) + (W / 2 if th < 1e-9 else (1 - math.cos(th)) / th ** 2 * W + (th - math.sin(th)) / th ** 3 * W @ W)
    return np.r_[w, np.linalg.solve(V, T[:3, 3])]


def _shift(c):
    return D.rigid(np.eye(3), c)


def exact(case, seed):
    kind = case["kind"]
    n64 = lambda a: a.detach().cpu().numpy()
    if kind in ("eval", "exact", "register"):
        *clouds, T0 = _single(case, seed)
        d = _Dense(*clouds, ISO_ELL[case["scene"]], 0.0 if case.get("dense") else CUTOFF)
        if kind == "register":
            return {"T": d.register(T0, 200, 1e-6)} if case["n_src"] <= 4000 else None
        f, g, M, Dg = d.eval(T0, kind == "exact")
        if kind == "exact":
            return {"f": n64(f), "g": n64(g), "H": n64(Dg + _gamma(g)), "D": n64(Dg), "n_pairs": None, "n_kept": None}
        return {"f": n64(f), "g": n64(g), "H": n64(_gamma(g) - M), "M": n64(M), "n_pairs": None, "n_kept": None}
    if kind == "cov":
        return [_covariances(x.float(), case["knn"], EIG_MAX["lidar" if case["scene"] == "mixed" else scene]).T.contiguous()
                for x, scene in _clouds(case, seed)]
    if kind == "clouds":
        if case["pairs"] > 1:
            return None
        scene, tx, tf, sx, sf, T0 = next(_cloud_pairs(case, seed))
        tc, sc = (_covariances(x, KNN, EIG_MAX[scene]).float() for x in (tx, sx))
        return {"T": _Dense(tx, tc, tf, sx, sc, sf, 0.0, CUTOFF).register(T0, 200, 1e-6)[None]}
    out, P, T, c, s = _net64(case, seed)
    if kind == "propose":
        tw = n64(out)
        T0 = [_shift(c[b]) @ _exp_se3(tw[b] * np.r_[1, 1, 1, s[b], s[b], s[b]]) @ _shift(-c[b]) for b in range(len(tw))]
        return {"twist": tw, "T0": np.stack(T0)}
    lab = np.stack([_log_se3(_shift(-c[b]) @ T[b] @ _shift(c[b])) / np.r_[1, 1, 1, s[b], s[b], s[b]] for b in range(len(c))])
    loss = ((out - _t(lab)) ** 2).sum(1).mean()
    loss.backward()
    return {"loss": n64(loss), "grad": n64(torch.cat([p.grad.reshape(-1) for p in P]))}
