"""Workloads of the library as a user's program runs them, for timing and for comparing results.

Every case calls the public Python entry points (``paper_2512_04996_gb300.vicp``) on clouds made on the GPU from a
seed, shaped like the library's own synthetic workloads: a sphere with a plane, a bumpy closed object with a 10:1
density gradient, and a depth-camera scene.  A case's fields:

  kind      step       one vicp_step on a grid that is already built (tracking a small scan against a kept model)
            frame      vicp_build_grid + vicp_dilate + vicp_correspond (a new target every frame, matches wanted)
            register   vicp_register, both clouds on the device
            register_host   vicp_register_host, both clouds in page-locked host memory
            offsets    vicp_offsets_static (voxel keys and offsets without allocating)
            batch      vicp_batch_build + vicp_batch_register of many pairs
            batch_host vicp_batch_register_host of many pairs
            loss       the differentiable loss of a batch, forward and backward
  cloud     sphere_plane, bumpy, scene; n target and m source points (batches: pairs, n_min, n_max; objects of even
            pairs are sphere_plane, of odd pairs bumpy)
  voxel / divisions   voxel edge, or the number of voxels along the longest side
  grid      fit (to the target at every build), keep (fitted once), explicit (given origin and dimensions)
  layers, iters, eps, rebuild, sparse, fp64   the library's parameters and flags
"""
import math

import numpy as np
import torch

from paper_2512_04996_gb300 import vicp

SCENE_BOX = ((-2.95, -2.45, 0.4), (6.05, 3.75, 4.85))   # corner and size of a box round every scene target


def _case(name, kind, **kw):
    d = dict(name=name, kind=kind, cloud="sphere_plane", n=0, m=0, voxel=0.0, divisions=0, layers=10, iters=1, eps=0.0,
             grid="keep", rebuild=False, sparse=False, fp64=False, pairs=0, n_min=0, n_max=0)
    d.update(kw)
    return d


def listed():
    return [
        # a small scan tracked against a model whose grid is kept: the smallest call, all latency
        _case("step_1k_on_4k", "step", n=4096, m=1000, divisions=64),
        # an object registered with a stopping rule and a grid fitted to it in the call (the plain way to use the library)
        _case("register_4k", "register", n=4096, m=4096, divisions=64, iters=30, eps=1e-5, grid="fit"),
        # a scanned object of the Stanford Bunny's size, clouds in host memory
        _case("register_host_40k", "register_host", cloud="bumpy", n=40000, m=40000, divisions=128, iters=50),
        # the benchmark scene: the whole registration with the grid rebuilt at every iteration
        _case("register_scene_226k", "register", cloud="scene", n=226000, m=226000, voxel=0.02, iters=30, rebuild=True),
        # a depth camera's frame against the one before it: build, dilate, match (ragged sizes: invalid pixels differ)
        _case("frame_scene_226k", "frame", cloud="scene", n=226000, m=221337, voxel=0.02),
        # the same on the sparse grid, for little memory
        _case("frame_sparse_226k", "frame", cloud="scene", n=226000, m=226000, voxel=0.02, sparse=True),
        # a high-resolution scan on a fixed map box of 1 cm voxels: the largest grid
        _case("frame_scene_1500k", "frame", cloud="scene", n=1500000, m=1500000, voxel=0.01, grid="explicit"),
        # one iteration at the method's stated precision (FP64 sums and solve)
        _case("step_fp64_226k", "step", cloud="scene", n=226000, m=226000, voxel=0.02, fp64=True),
        # voxel keys and offsets for a program that may not allocate
        _case("offsets_226k", "offsets", cloud="scene", n=226000, voxel=0.02, grid="explicit"),
        # a small batch of objects already on the device
        _case("batch_16_small", "batch", pairs=16, n_min=2000, n_max=8000, iters=40),
        # the batched workload: 256 uneven pairs from host memory
        _case("batch_host_256", "batch_host", pairs=256, n_min=2000, n_max=64000, iters=40),
        # a training step of the differentiable loss: 64 pairs of 20,000 points, gradients in poses and points
        _case("loss_64x20k", "loss", cloud="bumpy", pairs=64, n_min=20000, n_max=20000),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """Another case of the same ranges: sizes log-uniform from a thousand points to the largest listed, odd ones among
    them; object grids of 32 to 128 divisions; scene voxels that shrink with the resolution as the listed ones do."""
    kind = rng.choice(["step", "frame", "frame", "register", "register_host", "offsets", "batch", "batch_host", "loss"])
    c = dict(layers=rng.choice([6, 10, 10, 10, 15]))
    if kind in ("batch", "batch_host", "loss"):
        c["pairs"] = _log(rng, 2, 64)
        c["n_min"] = _log(rng, 1000, 8000)
        c["n_max"] = max(c["n_min"], _log(rng, 2000, 20000))
        c["iters"] = rng.randint(10, 40)
        c["cloud"] = "bumpy"
        c["fp64"] = kind != "loss" and rng.random() < 0.25
    else:
        scene = rng.random() < 0.5
        big = 1000000 if kind in ("step", "frame") else 226000
        c["cloud"] = "scene" if scene else rng.choice(["sphere_plane", "bumpy"])
        c["n"] = _log(rng, 20000 if scene else 1000, big if scene else 64000)
        c["m"] = max(1000, int(c["n"] * rng.uniform(0.5, 1.0))) if scene else c["n"]
        if scene:
            c["voxel"] = round(0.02 * math.sqrt(226000 / max(c["n"], 100000)), 4)
        else:
            c["divisions"] = rng.choice([32, 64, 100, 128])
        c["iters"] = rng.randint(5, 30)
        c["eps"] = rng.choice([0.0, 0.0, 1e-5])
        c["grid"] = "explicit" if kind == "offsets" else rng.choice(["fit", "keep", "keep"])
        c["rebuild"] = kind == "register" and rng.random() < 0.4
        c["sparse"] = kind == "frame" and rng.random() < 0.3
        c["fp64"] = kind != "offsets" and rng.random() < 0.2
        if kind == "offsets":
            c["cloud"] = "scene"
            c["divisions"] = 0
            c["voxel"] = round(rng.uniform(0.02, 0.06), 3)
    c = _case("", kind, **c)
    del c["name"]
    return c


# --- clouds ---------------------------------------------------------------------------------------------------------
def _gen(seed, salt=0):
    g = torch.Generator(device="cuda")
    g.manual_seed(1000003 * (int(seed) % (1 << 40)) + salt)
    return g


def _rand(g, *shape):
    return torch.rand(shape, generator=g, device="cuda", dtype=torch.float64)


def _unit(g, n):
    v = torch.randn((n, 3), generator=g, device="cuda", dtype=torch.float64)
    return v / v.norm(dim=1, keepdim=True)


def _rot(axis, angle):
    """Rodrigues' formula for (P, 3) unit axes and (P,) angles."""
    P = axis.shape[0]
    K = torch.zeros((P, 3, 3), dtype=torch.float64, device="cuda")
    K[:, 0, 1], K[:, 0, 2], K[:, 1, 2] = -axis[:, 2], axis[:, 1], -axis[:, 0]
    K = K - K.transpose(1, 2)
    eye = torch.eye(3, dtype=torch.float64, device="cuda")
    return eye + torch.sin(angle)[:, None, None] * K + (1 - torch.cos(angle))[:, None, None] * (K @ K)


def _motions(g, P, max_deg, max_trans):
    R = _rot(_unit(g, P), torch.deg2rad(max_deg * _rand(g, P)))
    t = _unit(g, P) * (max_trans * _rand(g, P) ** (1 / 3))[:, None]
    return R, t


def _xyzw(p):
    out = torch.zeros((p.shape[0], 4), dtype=torch.float32, device="cuda")
    out[:, :3] = p
    return out


def _objects(g, sizes, kinds, max_deg, max_trans):
    """Targets and sources (pooled, float64) of objects of the given sizes; kinds: True for bumpy ones.  A source is
    its target moved, with noise; a target's points come in no order, as a mesh's samples do."""
    P = len(sizes)
    n = torch.as_tensor(np.asarray(sizes), device="cuda")
    pair = torch.repeat_interleave(torch.arange(P, device="cuda"), n)
    N = int(pair.shape[0])
    first = torch.repeat_interleave(torch.cumsum(n, 0) - n, n)
    bumpy = torch.as_tensor(np.asarray(kinds), device="cuda")[pair]
    d = _unit(g, N)
    # bumpy: z with a density rising 10:1 from pole to pole, and a smooth random radius 1 +- 0.1
    u = _rand(g, N)
    z = (-0.55 + torch.sqrt(0.55 * 0.55 + 0.45 * (-0.65 + 2.2 * u))) / 0.45
    r = torch.sqrt(torch.clamp(1 - z * z, min=0.0))
    phi = 2 * math.pi * _rand(g, N)
    b = torch.stack([r * torch.cos(phi), r * torch.sin(phi), z], 1)
    K = 12
    w = _unit(g, P * K).reshape(P, K, 3) * (2 + 6 * _rand(g, P, K))[:, :, None]
    ph = 2 * math.pi * _rand(g, P, K)
    amp = torch.rand((P, K), generator=g, device="cuda", dtype=torch.float64)
    amp = 0.1 * amp / amp.sum(1, keepdim=True)
    rad = torch.ones(N, dtype=torch.float64, device="cuda")
    for k in range(K):
        rad += amp[pair, k] * torch.cos((b * w[pair, k]).sum(1) + ph[pair, k])
    # sphere + plane: the second half of the points on the 1 x 1 plane z = -1
    local = torch.arange(N, device="cuda") - first
    flat = local >= n[pair] // 2
    xy = _rand(g, N, 2) - 0.5
    plane = torch.cat([xy, torch.full((N, 1), -1.0, dtype=torch.float64, device="cuda")], 1)
    tgt = torch.where(bumpy[:, None], b * rad[:, None], torch.where(flat[:, None], plane, d))
    R, t = _motions(g, P, max_deg, max_trans)
    sigma = torch.where(bumpy, 0.002, 0.001)[:, None].double()
    src = torch.einsum("nij,nj->ni", R[pair], tgt) + t[pair]
    src = src + sigma * torch.randn((N, 3), generator=g, device="cuda", dtype=torch.float64)
    Rt = R.transpose(1, 2)
    T = torch.eye(4, dtype=torch.float64, device="cuda").repeat(P, 1, 1)
    T[:, :3, :3] = Rt
    T[:, :3, 3] = -(Rt @ t[:, :, None])[:, :, 0]
    return tgt, src, T


def _render(objs, boxes, res, R, t):
    """z-depth image of planes and boxes from a pinhole camera at (R, t), 640 x 480 scaled by res."""
    W, H, f = round(640 * res), round(480 * res), 525.0 * res
    u = torch.arange(W, device="cuda", dtype=torch.float64) - (319.5 * res)
    v = torch.arange(H, device="cuda", dtype=torch.float64) - (239.5 * res)
    ray = torch.stack([(u / f).expand(H, W), (v / f)[:, None].expand(H, W), torch.ones((H, W), device="cuda",
                       dtype=torch.float64)], -1).reshape(-1, 3)
    d = ray @ R.T
    best = torch.full((d.shape[0],), math.inf, dtype=torch.float64, device="cuda")
    for n, p in objs:
        s = ((p - t) @ n) / (d @ n)
        best = torch.minimum(best, torch.where(s > 1e-6, s, math.inf))
    for c, half, Rb in boxes:
        o, dl = (t - c) @ Rb, d @ Rb
        t1, t2 = (-half - o) / dl, (half - o) / dl
        lo, hi = torch.minimum(t1, t2).amax(1), torch.maximum(t1, t2).amin(1)
        hit = (hi >= lo) & (hi > 1e-6)
        best = torch.minimum(best, torch.where(hit, torch.where(lo > 1e-6, lo, hi), math.inf))
    return best, ray


def _scan(g, depth, ray, n, noise):
    """n pixels in scan order, chosen without replacement with weight 1/z^2 among the valid ones (depth 0.5 to 5.2 m,
    2% dropped), back-projected with depth noise."""
    z = depth
    ok = (z >= 0.5) & (z <= 5.2) & (_rand(g, z.shape[0]) >= 0.02)
    key = torch.where(ok, torch.log(_rand(g, z.shape[0])) * z * z, -math.inf)
    pick = torch.sort(torch.topk(key, n).indices).values
    zz = z[pick]
    if noise:
        zz = zz + noise * zz * zz * torch.randn(n, generator=g, device="cuda", dtype=torch.float64)
    return ray[pick] * zz[:, None]


def _scene(g, n, m):
    """Target and source scans of a room with boxes, cameras at most 5 degrees and 0.1 m apart."""
    c = torch.tensor
    f64 = dict(dtype=torch.float64, device="cuda")
    r = [float(x) for x in torch.rand(96, generator=g, device="cuda").tolist()]
    tilt = c([0.06 * r[0] - 0.03, 0.06 * r[1] - 0.03, -1.0], **f64)
    planes = [(tilt / tilt.norm(), c([0.0, 0.0, 4.8], **f64)), (c([0.0, -1.0, 0.0], **f64), c([0.0, 1.25, 0.0], **f64)),
              (c([1.0, 0.0, 0.2 * r[2] - 0.1], **f64), c([-2.7, 0.0, 0.0], **f64))]
    boxes = []
    eye = torch.eye(3, **f64)
    for k in range(9):
        q = r[5 + 8 * k:13 + 8 * k]
        size = [0.25 + 0.85 * q[i] for i in range(3)]
        yaw = _rot(c([[0.0, 1.0, 0.0]], **f64), c([0.5 * math.pi * q[5]], **f64))[0] if k % 2 else eye
        boxes.append((c([-2.2 + 4.6 * q[3], 1.25 - size[1] / 2, 1.2 + 3.1 * q[4]], **f64), c(size, **f64) / 2, yaw))
    for x, y, z, hs, a in ((0.5 * r[80] - 0.25, 0.3 * r[81] - 0.15, 0.55 + 0.15 * r[82], 0.12, r[83]),
                           (2 * r[84] - 1, 0.9 * r[85] - 0.6, 2 + r[86], 0.4, r[87])):
        boxes.append((c([x, y, z], **f64), c([hs, 0.8 * hs, 0.01], **f64),
                      _rot(_unit(g, 1), torch.deg2rad(c([10 + 30 * a], **f64)))[0]))
    res = math.sqrt(max(n, m) / 226000)
    R, t = _motions(g, 1, 5.0, 0.1)
    zero = torch.zeros(3, **f64)
    tgt = _scan(g, *_render(planes, boxes, res, eye, zero), n, 0.0)
    src = _scan(g, *_render(planes, boxes, res, R[0], t[0]), max(m, 1), 0.002)
    T = torch.eye(4, **f64)
    T[:3, :3], T[:3, 3] = R[0], t[0]
    return tgt, src, T


def _sizes(case):
    """Per-pair sizes of a batch, log-uniform in [n_min, n_max] (the same for every seed, as buffers are)."""
    r = np.random.RandomState(case["pairs"] + 7 * case["n_min"])
    lo, hi = math.log(case["n_min"]), math.log(case["n_max"])
    return np.round(np.exp(r.uniform(lo, hi, case["pairs"]))).astype(np.int32)


def _clouds(case, seed):
    g = _gen(seed)
    if case["pairs"]:
        n = _sizes(case)
        kinds = [case["cloud"] == "bumpy" or k % 2 == 1 for k in range(case["pairs"])]
        tgt, src, T = _objects(g, n, kinds, 15.0, 0.2 if case["kind"] != "loss" else 0.1)
        div = np.where(kinds, 128, 64).astype(np.int32)
        return dict(n=n, div=div, tgt=_xyzw(tgt), src=_xyzw(src), T=T)
    if case["cloud"] == "scene":
        tgt, src, T = _scene(g, case["n"], case["m"])
    else:
        bumpy = case["cloud"] == "bumpy"
        tgt, src, T = _objects(g, [case["n"]], [bumpy], 15.0 if bumpy else 10.0, 0.1 if bumpy else 0.05)
        T = T[0]
        if 0 < case["m"] < case["n"]:
            src = src[torch.randperm(case["n"], generator=g, device="cuda")[:case["m"]]]
    return dict(tgt=_xyzw(tgt), src=_xyzw(src), T=T)


def _explicit(case):
    """Origin and dimensions of the fixed map box."""
    o, size = SCENE_BOX
    return [float(np.float32(x)) for x in o], [int(math.ceil(s / case["voxel"])) for s in size]


def _start_pose(T):
    """A pose near the true one (a track from the frame before): the true motion with a tenth of it missing."""
    S = T.clone()
    S[..., :3, 3] *= 0.9
    return S.contiguous()


# --- the program ----------------------------------------------------------------------------------------------------
class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case = case
    c = _clouds(case, seed)
    kind = case["kind"]
    if kind in ("batch", "batch_host", "loss"):
        s.n, s.div = c["n"], c["div"]
        # shape 5: what the library's autotuner takes for the large batch; the default otherwise
        s.batch = vicp.Batch(dilation_layers=case["layers"], max_iters=case["iters"],
                             shape=5 if case["pairs"] >= 128 else -1,
                             flags=vicp.VICP_BATCH_FLAG_FP64 if case["fp64"] else 0)
        if kind == "batch_host":
            s.tgt_t, s.src_t = c["tgt"].cpu().pin_memory(), c["src"].cpu().pin_memory()
            s.tgt, s.src = s.tgt_t.numpy(), s.src_t.numpy()
        else:
            s.tgt, s.src = c["tgt"], c["src"]
        if kind == "loss":
            s.batch.build(s.tgt, s.n, None, s.div)
            s.T0 = c["T"].contiguous()
            g = _gen(seed, 1)
            s.xi = (0.02 * torch.randn((case["pairs"], 6), generator=g, device="cuda")).requires_grad_()
            s.src = s.src.requires_grad_()
            s.weight = 0.5 + torch.rand(case["pairs"], generator=g, device="cuda", dtype=torch.float64)
        return s
    flags = 0
    if case["grid"] == "keep":
        flags |= vicp.VICP_FLAG_KEEP_GRID
    for name, bit in (("rebuild", vicp.VICP_FLAG_REBUILD_EACH_ITER), ("sparse", vicp.VICP_FLAG_SPARSE_GRID),
                      ("fp64", vicp.VICP_FLAG_FP64_SOLVE)):
        if case[name]:
            flags |= bit
    kw = dict(voxel_size=case["voxel"], grid_divisions=case["divisions"], dilation_layers=case["layers"],
              max_iters=case["iters"], rmse_eps=case["eps"], flags=flags)
    if case["grid"] == "explicit":
        kw["origin"], kw["dims"] = _explicit(case)
    s.tgt, s.src = c["tgt"], c["src"]
    if kind == "offsets":
        s.grid = (kw["origin"], case["voxel"], kw["dims"])
        V = kw["dims"][0] * kw["dims"][1] * kw["dims"][2]
        s.keys = torch.empty(case["n"], dtype=torch.int32, device="cuda")
        s.offsets = torch.empty(V + 1, dtype=torch.int32, device="cuda")
        return s
    s.ctx = vicp.Context(**kw)
    if kind == "register_host":
        s.tgt_t, s.src_t = c["tgt"].cpu().pin_memory(), c["src"].cpu().pin_memory()
        s.tgt, s.src = s.tgt_t.numpy(), s.src_t.numpy()
    if kind in ("step", "frame"):
        s.pose0 = _start_pose(c["T"])
    if kind == "step":
        s.pose = s.pose0.clone()
        s.rmse = torch.zeros(1, dtype=torch.float64, device="cuda")
        s.ctx.build_grid(s.tgt)
        s.ctx.dilate()
    if kind == "frame":
        m = s.src.shape[0]
        s.nn = torch.empty(m, dtype=torch.int32, device="cuda")
        s.d2 = torch.empty(m, dtype=torch.float32, device="cuda")
        s.nfb = torch.zeros(1, dtype=torch.int32, device="cuda")
    return s


def run(s):
    kind = s.case["kind"]
    if kind == "step":
        s.pose.copy_(s.pose0)
        s.ctx.step(s.src, s.pose, s.rmse)
        return {"pose": s.pose, "rmse": s.rmse}
    if kind == "frame":
        s.ctx.build_grid(s.tgt)
        s.ctx.dilate()
        nn, d2, nfb = s.ctx.correspond(s.src, s.pose0, s.nn, s.d2, s.nfb)
        return {"nn": nn, "d2": d2, "fallbacks": nfb}
    if kind == "register":
        st, T, it, rmse = s.ctx.register(s.src, s.tgt)
        return {"status": st, "pose": T, "iterations": it, "rmse": rmse}
    if kind == "register_host":
        st, T, it, rmse = s.ctx.register_host(s.src, s.tgt)
        return {"status": st, "pose": T, "iterations": it, "rmse": rmse}
    if kind == "offsets":
        keys, off = vicp.vicp_offsets_static(s.tgt, *s.grid, s.keys, s.offsets)
        return {"keys": keys, "offsets": off}
    if kind == "batch":
        s.batch.build(s.tgt, s.n, None, s.div)
        st, T, it, rmse, each = s.batch.register(s.src, s.n)
        return {"status": st, "pose": T, "iterations": it, "rmse": rmse, "each": each}
    if kind == "batch_host":
        st, T, it, rmse, each = s.batch.register_host(s.src, s.n, s.tgt, s.n, None, s.div)
        return {"status": st, "pose": T, "iterations": it, "rmse": rmse, "each": each}
    loss = vicp.point_to_point_loss(s.xi, s.src, s.batch, s.n, s.T0)
    gx, gs = torch.autograd.grad((loss * s.weight).sum(), (s.xi, s.src))
    return {"loss": loss.detach(), "grad_xi": gx, "grad_src": gs}


def work(case):
    """Each cloud read once and each result written once; about 150 operations a source point and iteration
    (transform, quantise, eight candidates, the sums) and 30 a target point and build."""
    if case["pairs"]:
        n = int(_sizes(case).sum())
        its = case["iters"] if case["kind"] != "loss" else 1
        out = 20 * n if case["kind"] == "loss" else 152 * case["pairs"]
        return {"bytes": 32 * n + out, "flops": n * (150 * its + 30)}
    n, m = case["n"], case["m"]
    if case["kind"] == "offsets":
        V = math.prod(_explicit(case)[1])
        return {"bytes": 20 * n + 4 * V, "flops": 30 * n}
    if case["kind"] == "frame":
        return {"bytes": 16 * (n + m) + 8 * m, "flops": 30 * n + 150 * m}
    if case["kind"] == "step":
        return {"bytes": 16 * (n + m) + 256, "flops": 150 * m}
    builds = case["iters"] if case["rebuild"] else 1
    return {"bytes": 16 * (n + m) + 256, "flops": 30 * n * builds + 150 * m * case["iters"]}


# --- the same results from plain torch, sums and solves in 64 bits ------------------------------------------------------
# The method defines its decisions (voxel of a point, nearest candidate) on float32 coordinates with one rounding per
# operation, so those are made as it says; everything that is summed or solved is in float64.
_BIG = (1 << 31) - 1


def _f32(x):
    return torch.as_tensor(np.float32(x), device="cuda")


class _Exact:
    """The grid of one target: voxels, segments, root labels."""

    def __init__(self, tgt, case, divisions=None):
        q = tgt[:, :3].contiguous()
        if case["grid"] == "explicit":
            o, dims = _explicit(case)
            o = torch.tensor(o, dtype=torch.float32, device="cuda")
            h = np.float32(case["voxel"])
        else:
            o, hi = q.amin(0), q.amax(0)
            ext = hi - o
            div = case["divisions"] if divisions is None else divisions
            h = np.float32(case["voxel"]) if case["voxel"] > 0 else np.float32(float(ext.max())) / np.float32(div)
            inv = _f32(1.0 / float(h))
            dims = (torch.floor(ext * inv).long() + 1).tolist()
        self.q, self.o, self.dims, self.inv = q, o, dims, _f32(1.0 / float(h))
        keys = self.keys(q)
        self.all_keys = keys
        inside = torch.nonzero(keys >= 0)[:, 0]
        k, order = torch.sort(keys[inside], stable=True)
        self.ids, self.skeys = inside[order], k

    def keys(self, s):
        nx, ny, nz = self.dims
        c = (s - self.o) * self.inv
        top = torch.tensor([nx, ny, nz], dtype=torch.float32, device="cuda")
        ok = ((c >= 0) & (c < top)).all(1)
        i = torch.where(ok[:, None], torch.floor(c), 0.0).long()
        return torch.where(ok, i[:, 0] + nx * (i[:, 1] + ny * i[:, 2]), -1)

    def dilate(self, L):
        nx, ny, nz = self.dims
        lab = torch.full((nz * ny * nx,), _BIG, dtype=torch.int32, device="cuda")
        occ = torch.unique(self.skeys)
        lab[occ] = occ.int()
        lab = lab.view(nz, ny, nx)
        for _ in range(L):
            b = torch.full_like(lab, _BIG)
            for ax in range(3):
                n = lab.shape[ax]
                if n > 1:
                    b.narrow(ax, 1, n - 1).copy_(torch.minimum(b.narrow(ax, 1, n - 1), lab.narrow(ax, 0, n - 1)))
                    b.narrow(ax, 0, n - 1).copy_(torch.minimum(b.narrow(ax, 0, n - 1), lab.narrow(ax, 1, n - 1)))
            lab = torch.where(lab == _BIG, b, lab)
        self.lab = lab.reshape(-1)

    @staticmethod
    def _d2(a, b):
        d = a - b
        d = d * d
        return (d[..., 0] + d[..., 1]) + d[..., 2]

    def search(self, s):
        """Nearest target of each float32 point: in the root voxel, else over all points; ties to the smaller index."""
        v = self.keys(s)
        root = torch.where(v >= 0, self.lab[v.clamp(min=0)].long(), _BIG)
        nn = torch.empty(s.shape[0], dtype=torch.long, device="cuda")
        local = torch.nonzero(root < _BIG)[:, 0]
        for part in local.split(200000):
            a = torch.searchsorted(self.skeys, root[part])
            cnt = torch.searchsorted(self.skeys, root[part], right=True) - a
            qi = torch.repeat_interleave(torch.arange(part.shape[0], device="cuda"), cnt)
            k = torch.arange(qi.shape[0], device="cuda") - torch.repeat_interleave(torch.cumsum(cnt, 0) - cnt, cnt)
            j = self.ids[a[qi] + k]
            d = self._d2(s[part][qi], self.q[j])
            key = (d.view(torch.int32).long() << 32) | j
            best = torch.full((part.shape[0],), (1 << 63) - 1, dtype=torch.long, device="cuda")
            best.scatter_reduce_(0, qi, key, "amin")
            nn[part] = best & 0xffffffff
        far = torch.nonzero(root >= _BIG)[:, 0]
        idx = torch.arange(self.q.shape[0], device="cuda", dtype=torch.int32)
        x, y, z = (self.q[:, a].contiguous() for a in range(3))
        for part in far.split(max(1, (1 << 27) // self.q.shape[0])):
            p = s[part]
            d = (p[:, 0:1] - x).square_().add_((p[:, 1:2] - y).square_()).add_((p[:, 2:3] - z).square_())
            mn = d.amin(1, keepdim=True)
            nn[part] = torch.where(d == mn, idx, _BIG).amin(1).long()
        return nn, int(far.shape[0])


def _move32(T, src):
    """s_a = ((R_a0 x + R_a1 y) + R_a2 z) + t_a in float32, one rounding per operation."""
    P = T.float()
    x, y, z = (src[:, a].contiguous() for a in range(3))
    return torch.stack([((P[a, 0] * x + P[a, 1] * y) + P[a, 2] * z) + P[a, 3] for a in range(3)], 1)


def _update(T, s, q):
    """One rigid update (Kabsch, with the reflection rule) and the RMSE of the matches."""
    s, q = s.double(), q.double()
    rmse = torch.sqrt(((s - q) ** 2).sum(1).mean())
    cs, cq = s.mean(0), q.mean(0)
    H = ((s - cs).T @ (q - cq)).cpu().numpy()
    U, _, Vt = np.linalg.svd(H)
    D = np.diag([1.0, 1.0, np.sign(np.linalg.det(Vt.T @ U.T))])
    R = torch.from_numpy(Vt.T @ D @ U.T).cuda()
    dT = torch.eye(4, dtype=torch.float64, device="cuda")
    dT[:3, :3], dT[:3, 3] = R, cq - R @ cs
    return dT @ T, float(rmse)


def _register(grid, src, iters, eps):
    T, last, done = torch.eye(4, dtype=torch.float64, device="cuda"), None, 0
    rmse = 0.0
    for k in range(iters):
        s = _move32(T, src)
        nn, _ = grid.search(s)
        T, rmse = _update(T, s, grid.q[nn])
        done += 1
        if eps > 0 and last is not None and abs(rmse - last) < eps:
            break
        last = rmse
    return T, done, rmse


def _se3(xi):
    """Exp of one twist (translation part first), by the matrix exponential."""
    A = torch.zeros((4, 4), dtype=torch.float64, device="cuda")
    r, p = xi[:3], xi[3:]
    A = torch.stack([torch.stack([A[0, 0], -p[2], p[1], r[0]]), torch.stack([p[2], A[0, 0], -p[0], r[1]]),
                     torch.stack([-p[1], p[0], A[0, 0], r[2]]), A[3]])
    return torch.matrix_exp(A)


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch_host" and case["pairs"] > 64:
        return None   # minutes of brute force
    c = _clouds(case, seed)
    if case["pairs"]:
        n = c["n"]
        cut = np.concatenate([[0], np.cumsum(n)])
        poses, rmses, losses, gx, gs = [], [], [], [], []
        for k in range(case["pairs"]):
            tgt, src = c["tgt"][cut[k]:cut[k + 1]], c["src"][cut[k]:cut[k + 1]]
            grid = _Exact(tgt, case, int(c["div"][k]))
            grid.dilate(case["layers"])
            if kind != "loss":
                T, _, rmse = _register(grid, src, case["iters"], 0.0)
                poses.append(T.cpu().numpy())
                rmses.append(rmse)
                continue
            if k == 0:
                g = _gen(seed, 1)
                xi = (0.02 * torch.randn((case["pairs"], 6), generator=g, device="cuda")).double()
                w = 0.5 + torch.rand(case["pairs"], generator=g, device="cuda", dtype=torch.float64)
            x = xi[k].clone().requires_grad_()
            T = _se3(x) @ c["T"][k]
            nn, _ = grid.search(_move32(T.detach(), src))
            p = src[:, :3].double().requires_grad_()
            L = ((p @ T[:3, :3].T + T[:3, 3] - grid.q[nn].double()) ** 2).sum(1).mean()
            dx, dp = torch.autograd.grad(w[k] * L, (x, p))
            losses.append(L.detach())
            gx.append(dx)
            gs.append(torch.cat([dp, torch.zeros_like(dp[:, :1])], 1))
        if kind == "loss":
            return {"loss": torch.stack(losses), "grad_xi": torch.stack(gx), "grad_src": torch.cat(gs)}
        return {"status": None, "pose": np.stack(poses), "iterations": None, "rmse": np.array(rmses), "each": None}
    if kind == "offsets":
        return None   # whole numbers
    grid = _Exact(c["tgt"], case)
    grid.dilate(case["layers"])
    if kind == "frame":
        T = _start_pose(c["T"])
        s = _move32(T, c["src"])
        nn, _ = grid.search(s)
        s64 = c["src"][:, :3].double() @ T[:3, :3].T + T[:3, 3]
        return {"nn": None, "d2": ((s64 - grid.q[nn].double()) ** 2).sum(1), "fallbacks": None}
    if kind == "step":
        T = _start_pose(c["T"])
        s = _move32(T, c["src"])
        nn, _ = grid.search(s)
        T, rmse = _update(T, s, grid.q[nn])
        return {"pose": T, "rmse": torch.tensor([rmse], dtype=torch.float64)}
    T, _, rmse = _register(grid, c["src"], case["iters"], case["eps"])
    return {"status": None, "pose": T.cpu().numpy(), "iterations": None, "rmse": rmse}
