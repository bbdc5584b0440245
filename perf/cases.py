"""The work that a user of this framework has it do, as measurable cases.

Every case is one call, or one step of a program, through the package's public
entry points: novel-view renders, optimisation steps (forward, loss,
backward), batches of scenes, spatially varying absorption, the BVH build with
arbitrary ray queries, the mesh update after a gradient, and the image losses.
Sizes span what the repository's own benchmark and tests use, from a 64x64
frame of an icosphere to a million-triangle optimisation step.

A case's "kind" names the step; the other values are its sizes and options.
All inputs come from the seed: the mesh's vertices are displaced by seeded
noise, and materials, cameras, environments, targets and textures are drawn
from it.
"""
import functools
import math

import numpy as np
import torch

import paper_2603_00413_gb300 as dt
from paper_2603_00413_gb300 import scenes as S

DEV = "cuda"


def listed():
    return [
        # one frame of the smallest scene (interactive preview, a 64x64 request): launches and latency
        {"name": "frame_64", "kind": "frame", "mesh": "ico", "n": 3, "views": 1, "w": 64, "h": 64, "depth": 4, "spp": 1},
        # novel views of a trained object at inference depth 8, an image size that no tile divides
        {"name": "novel_views", "kind": "frame", "mesh": "tori", "n": 72, "views": 12, "w": 509, "h": 383, "depth": 8, "spp": 1},
        # the main optimisation step: normals, refit, forward, L2 loss, backward over many views
        {"name": "train_step", "kind": "train", "mesh": "tori", "n": 72, "views": 48, "w": 512, "h": 512, "depth": 8, "spp": 1, "ckpt": False, "env": 64},
        # the same step through autograd on a small mesh at the training depth 4, BVH built in the call
        {"name": "autograd_small", "kind": "autograd", "mesh": "ico", "n": 4, "views": 2, "w": 96, "h": 72, "depth": 4, "spp": 1},
        # the largest step: a million triangles, depth 16, jittered samples, checkpointed tape, BVH rebuilt
        {"name": "large_step", "kind": "train", "mesh": "bumpy", "n": 300, "views": 1, "w": 800, "h": 800, "depth": 16, "spp": 8, "ckpt": True, "env": 1024},
        # many scenes of uneven size in one set of launches (dataset training, a server's batch)
        {"name": "batch_scenes", "kind": "batch", "scenes": 40, "faces_lo": 2000, "faces_hi": 200000, "side_lo": 128, "side_hi": 640, "depth": 12},
        # spatially varying absorption on a dense grid, moments tape, with the environment's gradient
        {"name": "absorption_grid", "kind": "medium", "mesh": "tori", "n": 72, "views": 16, "w": 384, "h": 384, "depth": 8, "spp": 1, "levels": 0, "nodes": 64, "moments": True},
        # absorption as a multi-resolution hash texture, full tape
        {"name": "absorption_hash", "kind": "medium", "mesh": "tori", "n": 72, "views": 8, "w": 360, "h": 360, "depth": 8, "spp": 1, "levels": 8, "nodes": 128, "moments": False},
        # a mesh loaded or remeshed: BVH built, then closest hits of arbitrary rays
        {"name": "build_query", "kind": "query", "mesh": "bumpy", "n": 100, "rays": 200001},
        # the mesh update after a gradient: two smoothing solves and AdamUniform
        {"name": "mesh_update", "kind": "update", "mesh": "bumpy", "n": 110, "iters": 100},
        # the edge regulariser of a mesh just remeshed: its topology is built in the call
        {"name": "edge_loss", "kind": "edge", "mesh": "bumpy", "n": 150},
        # the colour and tone losses over a batch of rendered views
        {"name": "image_losses", "kind": "loss", "pixels": 6291456},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["frame", "frame", "train", "train", "autograd", "batch", "medium", "medium", "query", "update", "edge", "loss"])
    if kind == "loss":
        return {"kind": kind, "pixels": _log(rng, 4000, 26000000)}
    if kind == "batch":
        return {"kind": kind, "scenes": _log(rng, 2, 40), "faces_lo": 2000, "faces_hi": 200000, "side_lo": 128,
                "side_hi": _log(rng, 200, 640), "depth": rng.randint(4, 12)}
    if kind in ("query", "update", "edge"):
        c = {"kind": kind, "mesh": "bumpy", "n": _log(rng, 15, 300)}
        if kind == "query":
            c["rays"] = _log(rng, 1000, 1000000)
        if kind == "update":
            c["iters"] = rng.choice([60, 100])
        return c
    mesh = rng.choice(["ico", "tori", "bumpy"])
    n = {"ico": lambda: rng.randint(3, 5), "tori": lambda: _log(rng, 32, 96), "bumpy": lambda: _log(rng, 15, 200)}[mesh]()
    c = {"kind": kind, "mesh": mesh, "n": n, "depth": rng.choice([4, 4, 6, 8, 8]), "spp": rng.choice([1, 1, 1, 2, 4])}
    if kind == "autograd":
        return dict(c, mesh="ico", n=rng.randint(3, 4), views=1, w=rng.randint(32, 110), h=rng.randint(32, 90), depth=4, spp=1)
    # camera rays of the whole case, then their split over views and an uneven image
    rays = _log(rng, 4096, {"frame": 8000000, "train": 8000000, "medium": 800000}[kind])
    side = min(_log(rng, 48, 800), int(math.sqrt(rays / c["spp"])))
    c["w"] = max(16, int(side * rng.uniform(0.8, 1.25)))
    c["h"] = max(16, int(side * rng.uniform(0.8, 1.25)))
    c["views"] = max(1, rays // (c["w"] * c["h"] * c["spp"]))
    if kind == "train":
        c["ckpt"] = rng.random() < 0.4
        c["env"] = rng.choice([64, 256, 1024])
    if kind == "medium":
        c["levels"] = rng.choice([0, 4, 8])
        c["nodes"] = rng.choice([32, 64, 100]) if c["levels"] == 0 else 128
        c["moments"] = rng.random() < 0.5
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _bumpy_sphere(n):
    """A closed sphere of 12 n^2 triangles (a cube's n x n faces pushed onto
    the sphere) with bumps of three octaves of amplitude 0.1."""
    i, j = np.meshgrid(np.arange(n), np.arange(n), indexing="ij")
    quads = []
    for axis in range(3):
        u, v = (axis + 1) % 3, (axis + 2) % 3
        for side in (0, n):
            q = np.zeros((n, n, 4, 3), np.int64)
            for c, (di, dj) in enumerate(((0, 0), (1, 0), (1, 1), (0, 1))):
                q[:, :, c, axis], q[:, :, c, u], q[:, :, c, v] = side, i + di, j + dj
            quads.append((q if side else q[:, :, ::-1]).reshape(-1, 4, 3))
    q = np.concatenate(quads)
    key = (q[..., 0] * (n + 1) + q[..., 1]) * (n + 1) + q[..., 2]
    ids, idx = np.unique(key.reshape(-1), return_inverse=True)
    idx = idx.reshape(-1, 4)
    P = np.stack([ids // (n + 1) ** 2, ids // (n + 1) % (n + 1), ids % (n + 1)], 1) * (2.0 / n) - 1.0
    P = np.tan(P * (math.pi / 4))  # near-equal cells
    P /= np.linalg.norm(P, axis=1, keepdims=True)
    r = np.ones(len(P))
    for o in range(3):
        a = np.random.default_rng(o).normal(size=(6, 3))
        r += 0.1 * 0.5 ** o * np.sin(P @ a.T * (3.0 * 2 ** o)).mean(1)
    P *= (r / r.max())[:, None]
    return P.astype(np.float32), np.concatenate([idx[:, [0, 1, 2]], idx[:, [0, 2, 3]]]).astype(np.int32)


@functools.lru_cache(maxsize=64)
def _mesh(kind, n):
    """A base mesh (the same for every seed): vertices and faces."""
    if kind == "ico":
        return S.icosphere(n)
    if kind == "tori":
        return S.two_tori_mesh(n)
    return _bumpy_sphere(n)


def _geometry(kind, n, rng):
    """The base mesh with vertices displaced by a tenth of the mean edge."""
    V, F = _mesh(kind, n)
    edge = float(np.mean(np.linalg.norm(V[F[:4096, 0]] - V[F[:4096, 1]], axis=1)))
    V = (V + rng.normal(0.0, 0.05 * edge, size=V.shape)).astype(np.float32)
    return V, F


def _to(x):
    return torch.from_numpy(np.ascontiguousarray(x)).to(DEV)


def _scene_arrays(c, seed):
    """Host arrays of a scene: geometry, materials, environment, cameras."""
    rng = np.random.default_rng(seed)
    V, F = _geometry(c["mesh"], c["n"], rng)
    env_w = c.get("env", 64)
    env = S.sh_env_map(min(env_w, 256), min(env_w, 256) // 2, seed)
    if env_w > 256:  # a photograph's resolution: the smooth field upsampled, with texel noise
        k = env_w // 256
        env = np.repeat(np.repeat(env, k, 0), k, 1) * rng.uniform(0.9, 1.1, (env_w // 2, env_w, 1))
    rot = np.linalg.qr(rng.normal(size=(3, 3)))[0]
    cams = np.stack([v.as_array() for v in S.fibonacci_views(c["views"], 3.0, c["w"], c["h"])])
    cams[:, :3] = cams[:, :3] @ rot.T
    return dict(V=V, F=F, ior=np.float32([rng.uniform(1.3, 1.7)]), sigma=rng.uniform(0.0, 2.0, 3).astype(np.float32),
                env=env.astype(np.float32), cams=cams.astype(np.float32))


def _params(c, seed, moments=False):
    return dt.Params(c["depth"], spp=c["spp"], jitter=1 if c["spp"] > 1 else 0, seed=seed,
                     checkpoint=bool(c.get("ckpt")), moments=moments)


def _scene(c, seed, moments=False):
    s = {k: _to(v) for k, v in _scene_arrays(c, seed).items()}
    s["N"] = dt.vertex_normals(s["V"], s["F"])
    s["bvh"] = dt.build_bvh(s["V"], s["F"])
    s["params"] = _params(c, seed, moments)
    rays = c["views"] * c["w"] * c["h"] * c["spp"]
    cap = int(rays * min(2 * c["depth"] + 3, 14)) + 4096
    s["ws"] = dt.Workspace(cap, DEV, level_capacity=2 * rays if c.get("ckpt") else 0, moments=moments)
    return s


def _target(c, s, seed, sigma):
    """The image that an optimisation aims at: the render of displaced vertices."""
    g = torch.Generator(DEV).manual_seed(seed)
    Vt = s["V"] + sigma * torch.randn(s["V"].shape, generator=g, device=DEV)
    bvh = dt.build_bvh(Vt, s["F"])
    img, _ = dt.render(Vt, s["F"], bvh, dt.vertex_normals(Vt, s["F"]), s["ior"], s["sigma"], s["env"], s["cams"],
                       c["w"], c["h"], s["params"], ws=s["ws"])
    return img


def _batch_specs(c, seed):
    """Faces, image side, depth and seed of every scene of a batch (sizes from
    the case alone, spread over their logarithm; contents from the seed)."""
    rng = np.random.default_rng(c["scenes"])
    out = []
    for i in range(c["scenes"]):
        faces = math.exp(rng.uniform(math.log(c["faces_lo"]), math.log(c["faces_hi"])))
        side = int(round(math.exp(rng.uniform(math.log(c["side_lo"]), math.log(c["side_hi"])))))
        mesh = "tori" if rng.uniform() < 0.3 else "bumpy"
        n = round(math.sqrt(faces / (12.0 if mesh == "bumpy" else 10.1)))
        out.append({"mesh": mesh, "n": max(14, min(n, 130)), "views": 1, "w": side, "h": side, "spp": 1,
                    "depth": int(rng.integers(4, c["depth"] + 1)), "seed": 1000 * seed + i})
    return out


def prepare(case, seed):
    c, kind = case, case["kind"]
    g = torch.Generator(DEV).manual_seed(seed)
    s = {"case": c}
    if kind == "loss":
        n = c["pixels"]
        target = torch.rand(n, 3, generator=g, device=DEV) * 1.5
        s["img"] = (target + 0.1 * torch.randn(n, 3, generator=g, device=DEV)).clamp_(min=0.0)
        s["target"] = target
        s["grad"], s["loss"] = torch.empty_like(target), torch.empty(3, device=DEV)
        return s
    if kind in ("query", "update", "edge"):
        V, F = _geometry(c["mesh"], c["n"], np.random.default_rng(seed))
        s["V"], s["F"] = _to(V), _to(F)
        if kind == "query":
            o = torch.randn(c["rays"], 3, generator=g, device=DEV)
            s["o"] = 2.0 * o / o.norm(dim=1, keepdim=True)
            d = 0.5 * torch.randn(c["rays"], 3, generator=g, device=DEV) - s["o"]
            s["d"] = d / d.norm(dim=1, keepdim=True)
        if kind == "update":
            s["opt"] = dt.LargeStepsOptimizer(s["V"], s["F"], iters=c["iters"])
            # an image gradient: smooth over the surface, with per-vertex noise
            s["g"] = (torch.sin(4.0 * s["V"]) + 0.5 * torch.randn(s["V"].shape, generator=g, device=DEV)) * 1e-4
        return s
    if kind == "batch":
        specs = _batch_specs(c, seed)
        sizes = [b["w"] * b["h"] for b in specs]
        s["img"] = torch.empty(3 * sum(sizes), device=DEV)
        s["outs"], items, at = [], [], 0
        for b, n in zip(specs, sizes):
            a = {k: _to(v) for k, v in _scene_arrays(b, b["seed"]).items()}
            items.append(dt.BatchItem(a["V"], a["F"], dt.build_bvh(a["V"], a["F"]), dt.vertex_normals(a["V"], a["F"]),
                                      a["ior"], a["sigma"], a["env"], a["cams"], b["w"], b["h"], dt.Params(b["depth"])))
            s["outs"].append(s["img"][at:at + 3 * n].view(1, b["h"], b["w"], 3))
            at += 3 * n
        s["items"] = items
        s["target"] = torch.rand(3 * sum(sizes), generator=g, device=DEV) * 1.5
        s["grad"] = torch.empty_like(s["img"])
        s["grads"] = [s["grad"].as_strided(o.shape, o.stride(), o.storage_offset()) for o in s["outs"]]
        s["dV"] = torch.empty(sum(i.V.shape[0] for i in items), 3, device=DEV)
        s["dmat"] = torch.empty(len(items), 4, device=DEV)
        dVs = s["dV"].split([i.V.shape[0] for i in items])
        s["gouts"] = [(v, m[:1], m[1:]) for v, m in zip(dVs, s["dmat"])]
        s["ws"] = dt.Workspace(16 * sum(sizes) + 4096, DEV)
        return s
    if kind == "autograd":
        s.update({k: _to(v) for k, v in _scene_arrays(c, seed).items()})
        for k in ("V", "ior", "sigma"):
            s[k].requires_grad_(True)
        s["params"] = _params(c, seed)
        s["g"] = torch.rand(c["views"], c["h"], c["w"], 3, generator=g, device=DEV)
        return s
    s.update(_scene(c, seed, bool(c.get("moments"))))
    if kind == "frame":
        s["out"] = torch.empty(c["views"], c["h"], c["w"], 3, device=DEV)
        return s
    if kind == "train":
        s["target"] = _target(c, s, seed, 0.002)
        return s
    lo, hi = (-1.25,) * 3, (1.25,) * 3
    step = 0.5 * 2.5 / (c["nodes"] - 1)
    if c["levels"]:
        res = S.hash_texture_resolutions(c["levels"], 16, c["nodes"])
        table = torch.rand(c["levels"], 1 << 19, 3, generator=g, device=DEV) * (2.0 / c["levels"])
        s["medium"] = dt.HashTexture(table, res, lo, hi, step)
    else:
        coarse = torch.randn(1, 3, 9, 9, 9, generator=g, device=DEV)
        mu = torch.nn.functional.interpolate(coarse, size=(c["nodes"],) * 3, mode="trilinear", align_corners=True)
        s["medium"] = dt.Medium(torch.nn.functional.softplus(2.0 * mu - 0.5)[0].permute(1, 2, 3, 0).contiguous(), lo, hi, step)
    s["g"] = torch.rand(c["views"], c["h"], c["w"], 3, generator=g, device=DEV)
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------
def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "loss":
        return dt.paper_loss_grad(s["img"], s["target"], 1.0, 0.5, grad=s["grad"], loss=s["loss"])
    if kind == "query":
        bvh = dt.build_bvh(s["V"], s["F"])
        return dt.closest_hit(bvh, s["o"], s["d"])
    if kind == "update":
        V = s["opt"].step(s["g"])
        return V, s["opt"].state[: 4 * V.numel()].view(torch.float32)  # vertices and first moment
    if kind == "edge":
        return dt.edge_loss_grad(s["V"], s["F"])
    if kind == "batch":
        _, tape = dt.render_batch(s["items"], ws=s["ws"], outs=s["outs"])
        _, loss = dt.l2_loss_grad(s["img"], s["target"], grad=s["grad"])
        dt.render_batch_backward(tape, s["grads"], outs=s["gouts"])
        return s["img"], loss, s["dV"], s["dmat"]
    if kind == "autograd":
        leaves = [s[k] for k in ("V", "ior", "sigma")]
        for x in leaves:
            x.grad = None
        img = dt.render_differentiable(leaves[0], s["F"], leaves[1], leaves[2], s["env"], s["cams"], c["w"], c["h"], s["params"])
        (img * s["g"]).sum().backward()
        return [img] + [x.grad for x in leaves]
    args = (s["ior"], s["sigma"], s["env"], s["cams"], c["w"], c["h"], s["params"])
    if kind == "frame":
        img, _ = dt.render(s["V"], s["F"], s["bvh"], s["N"], *args, ws=s["ws"], out=s["out"], check=False)
        return img
    if kind == "train":
        N = dt.vertex_normals(s["V"], s["F"])
        if c["ckpt"]:
            s["bvh"].build(s["V"], s["F"])
        else:
            dt.refit_bvh(s["bvh"], s["V"], s["F"])
        img, tape = dt.render(s["V"], s["F"], s["bvh"], N, *args, ws=s["ws"])
        grad, loss = dt.l2_loss_grad(img, s["target"])
        return (img, loss) + dt.render_backward(tape, grad)
    img, tape = dt.render(s["V"], s["F"], s["bvh"], s["N"], *args, ws=s["ws"], medium=s["medium"])
    return (img,) + dt.render_backward(tape, s["g"], env_grad=True)


# ---------------------------------------------------------------------------
# the least that a pass has to move and compute
# ---------------------------------------------------------------------------
SEGMENTS_PER_RAY = 4.5  # about half of the camera rays hit; a hit ray's tree adds some 2 D segments
SEGMENT_FLOPS = 1500.0  # a search of some 25 tree nodes, three triangle tests, the optics of one hit


def _faces(c):
    return {"ico": lambda n: 20 * 4 ** n, "tori": lambda n: int(10.1 * n * n), "bumpy": lambda n: 12 * n * n}[c["mesh"]](c["n"])


def work(case):
    c, kind = case, case["kind"]
    if kind == "loss":  # two images read, a gradient written
        return {"bytes": 36.0 * c["pixels"], "flops": 60.0 * c["pixels"]}
    if kind == "batch":
        each = [work(dict(b, kind="train", ckpt=False)) for b in _batch_specs(c, 0)]
        return {k: sum(w[k] for w in each) for k in ("bytes", "flops")}
    nf = _faces(c)
    nv = nf // 2
    mesh = 12.0 * nf + 12.0 * nv
    if kind == "query":  # mesh and rays read, hits written
        return {"bytes": mesh + 40.0 * c["rays"], "flops": 100.0 * nf * max(1.0, math.log2(nf)) + SEGMENT_FLOPS * c["rays"]}
    if kind == "update":  # per iteration one pass over the neighbour list and the five vectors
        return {"bytes": 24.0 * nv + 24.0 * nv * 3, "flops": 2.0 * c["iters"] * nv * 60.0}
    if kind == "edge":  # mesh read, gradient written
        return {"bytes": mesh + 12.0 * nv, "flops": 300.0 * nf}
    rays = float(c["views"] * c["w"] * c["h"] * c["spp"])
    img = 12.0 * rays / c["spp"]
    seg = SEGMENTS_PER_RAY * rays
    if kind == "frame":
        return {"bytes": mesh + 12.0 * nv + img, "flops": seg * SEGMENT_FLOPS}
    # target or seed read, image and vertex gradient written; the backward about as much arithmetic as the optics
    w = {"bytes": mesh + 12.0 * nv + 2.0 * img, "flops": seg * (SEGMENT_FLOPS + 600.0)}
    if kind == "medium":  # the field read and its gradient written; half of the segments run inside, some 15 samples each
        samples = 0.5 * seg * 15.0 * (c["nodes"] / 128.0) * max(1, c["levels"])
        w["bytes"] += 28.0 * (c["levels"] * (1 << 19) if c["levels"] else c["nodes"] ** 3)
        w["flops"] += samples * 100.0
    return w


# ---------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ---------------------------------------------------------------------------
def _dev64():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _normals64(V, F):
    e1, e2 = V[F[:, 1]] - V[F[:, 0]], V[F[:, 2]] - V[F[:, 0]]
    c = torch.linalg.cross(e1, e2)
    u = c / c.norm(dim=1, keepdim=True)
    N = torch.zeros_like(V)
    for k in range(3):
        N = N.index_add(0, F[:, k], u)
    return N / 3.0


@torch.no_grad()
def _closest64(V, F, o, d, src, t_min):
    """Closest hit of every ray by testing every triangle: triangle or -1."""
    v0, e1, e2 = V[F[:, 0]], V[F[:, 1]] - V[F[:, 0]], V[F[:, 2]] - V[F[:, 0]]
    out = []
    step = max(1, 24_000_000 // len(F))
    ids = torch.arange(len(F), device=V.device)
    for a in range(0, len(o), step):
        O, D = o[a:a + step, None], d[a:a + step, None]
        p = torch.linalg.cross(D, e2[None].expand(len(D), -1, -1))
        inv = 1.0 / (e1 * p).sum(-1)
        s = O - v0
        b1 = (s * p).sum(-1) * inv
        q = torch.linalg.cross(s, e1[None].expand(len(D), -1, -1))
        b2 = (D * q).sum(-1) * inv
        t = (e2 * q).sum(-1) * inv
        ok = (t > t_min) & (b1 >= 0) & (b2 >= 0) & (b1 + b2 <= 1) & (ids != src[a:a + step, None])
        t = torch.where(ok, t, math.inf)
        best, tri = t.min(1)
        out.append(torch.where(best < math.inf, tri, -1))
    return torch.cat(out)


def _hit64(V, F, o, d, tri):
    v0, v1, v2 = (V[F[tri, k]] for k in range(3))
    e1, e2 = v1 - v0, v2 - v0
    p = torch.linalg.cross(d, e2)
    det = (e1 * p).sum(-1)
    s = o - v0
    q = torch.linalg.cross(s, e1)
    return (e2 * q).sum(-1) / det, (s * p).sum(-1) / det, (d * q).sum(-1) / det, torch.linalg.cross(e1, e2)


def _env64(env, d):
    h, w = env.shape[:2]
    phi = torch.atan2(d[:, 2], d[:, 0])
    phi = torch.where(phi < 0, phi + 2 * math.pi, phi)
    u = phi / (2 * math.pi) * w - 0.5
    v = torch.acos(d[:, 1].clamp(-1, 1)) / math.pi * h - 0.5
    x, y = u.detach().floor(), v.detach().floor()
    ax, ay = (u - x)[:, None], (v - y)[:, None]
    x0, x1 = x.long() % w, (x.long() + 1) % w
    y0, y1 = y.long().clamp(0, h - 1), (y.long() + 1).clamp(0, h - 1)
    return (env[y0, x0] * (1 - ax) + env[y0, x1] * ax) * (1 - ay) + (env[y1, x0] * (1 - ax) + env[y1, x1] * ax) * ay


def _render64(c, a, t_min):
    """The image of a scene (1 sample at pixel centres), level by level; differentiable at fixed hits."""
    V, F, env, w, h = a["V"], a["F"].long(), a["env"], c["w"], c["h"]
    N = _normals64(V, F)
    cam = a["cams"]
    f = torch.nn.functional.normalize(cam[:, 3:6] - cam[:, :3], dim=1)
    r = torch.nn.functional.normalize(torch.linalg.cross(f, cam[:, 6:9]), dim=1)
    u = torch.linalg.cross(r, f)
    th = torch.tan(0.5 * cam[:, 9] * math.pi / 180.0)
    px = (2.0 * (torch.arange(w, device=V.device) + 0.5) / w - 1.0) * (w / h)
    py = 1.0 - 2.0 * (torch.arange(h, device=V.device) + 0.5) / h
    d = (f[:, None, None] + r[:, None, None] * (px[None, None, :, None] * th[:, None, None, None])
         + u[:, None, None] * (py[None, :, None, None] * th[:, None, None, None])).reshape(-1, 3)
    d = torch.nn.functional.normalize(d, dim=1)
    o = cam[:, None, :3].expand(-1, w * h, -1).reshape(-1, 3)
    pix = torch.arange(len(o), device=V.device)
    W = torch.ones(len(o), 3, dtype=V.dtype, device=V.device)
    src = torch.full((len(o),), -1, device=V.device)
    img = torch.zeros(len(o), 3, dtype=V.dtype, device=V.device)
    for k in range(c["depth"] + 1):
        tri = _closest64(V, F, o.detach(), d.detach(), src, t_min)
        m = tri < 0
        img = img.index_add(0, pix[m], W[m] * _env64(env, d[m]))
        if k == c["depth"] or m.all():
            break
        o, d, W, pix, tri = o[~m], d[~m], W[~m], pix[~m], tri[~m]
        t, b1, b2, ng = _hit64(V, F, o, d, tri)
        enter = (d * ng).sum(-1) < 0
        x = o + d * t[:, None]
        mm = N[F[tri, 0]] * (1 - b1 - b2)[:, None] + N[F[tri, 1]] * b1[:, None] + N[F[tri, 2]] * b2[:, None]
        n = mm / mm.norm(dim=1, keepdim=True)
        ns = torch.where(enter[:, None], n, -n)
        cos = -(d * ns).sum(-1)
        A = torch.where(enter[:, None], torch.ones_like(W), torch.exp(-a["sigma"] * t[:, None]))
        one = torch.ones_like(cos)
        e1, e2 = torch.where(enter, one, a["ior"] * one), torch.where(enter, a["ior"] * one, one)
        eta = e2 / e1
        kappa = eta * eta - (1 - cos * cos)
        tir = kappa < 0
        ct = torch.sqrt(torch.where(tir, one, kappa)) / eta
        rs = (e1 * cos - e2 * ct) / (e1 * cos + e2 * ct)
        rp = (e1 * ct - e2 * cos) / (e1 * ct + e2 * cos)
        R = torch.where(tir, one, 0.5 * (rs * rs + rp * rp))
        wr = 2 * cos[:, None] * ns + d
        wt = (d + cos[:, None] * ns) / eta[:, None] - ct[:, None] * ns
        good = cos > 0
        two = good & ~tir
        WA = W * A
        o = torch.cat([x[good], x[two]])
        d = torch.cat([wr[good], wt[two]])
        W = torch.cat([(WA * R[:, None])[good], (WA * (1 - R)[:, None])[two]])
        pix = torch.cat([pix[good], pix[two]])
        src = torch.cat([tri[good], tri[two]])
    return img.reshape(c["views"], h, w, 3)


def _laplacian64(F, nv):
    e = torch.cat([F[:, [0, 1]], F[:, [1, 2]], F[:, [2, 0]]])
    e = torch.cat([e, e.flip(1)])
    e = torch.unique(e[:, 0] * nv + e[:, 1])
    i, j = e // nv, e % nv
    deg = torch.zeros(nv, dtype=torch.float64, device=F.device).index_add(0, i, torch.ones(len(i), dtype=torch.float64, device=F.device))
    return i, j, deg


def _solve64(i, j, deg, lam, b):
    """(I + lam L) x = b by conjugate gradients to 1e-13."""
    apply = lambda x: x + lam * (deg[:, None] * x - torch.zeros_like(x).index_add(0, i, x[j]))  # noqa: E731
    x = torch.zeros_like(b)
    r = b.clone()
    p, rr = r.clone(), (r * r).sum(0)
    r0 = rr.clone()
    for _ in range(400):
        ap = apply(p)
        al = rr / (p * ap).sum(0)
        x, r = x + al * p, r - al * ap
        new = (r * r).sum(0)
        if bool((new < 1e-26 * r0).all()):
            break
        p, rr = r + new / rr * p, new
    return x


def exact(case, seed):
    c, kind = case, case["kind"]
    brute = kind in ("frame", "autograd") and c["spp"] == 1 and c["views"] * c["w"] * c["h"] * _faces(c) < 1.5e8
    if not (brute or kind in ("loss", "update", "edge")) and not (kind == "query" and c["rays"] * _faces(c) < 2.5e10):
        return None  # a search of every triangle for every segment would take minutes
    f64 = lambda x: x.to(_dev64(), torch.float64)  # noqa: E731
    if brute:
        a = {k: f64(torch.from_numpy(v)) for k, v in _scene_arrays(c, seed).items()}
        t_min = float(np.float32(1e-5))
        if kind == "frame":
            with torch.no_grad():
                return _render64(c, a, t_min)
        leaves = [a[k].requires_grad_(True) for k in ("V", "ior", "sigma")]
        img = _render64(c, a, t_min)
        g = torch.rand(c["views"], c["h"], c["w"], 3, generator=torch.Generator(DEV).manual_seed(seed), device=DEV)
        return [img.detach()] + list(torch.autograd.grad((img * f64(g)).sum(), leaves))
    s = prepare(case, seed)
    if kind == "query":
        V, F, o, d = f64(s["V"]), s["F"].long().to(_dev64()), f64(s["o"]), f64(s["d"])
        tri = _closest64(V, F, o, d, torch.full((len(o),), -1, device=V.device), float(np.float32(1e-5)))
        t, b1, b2, _ = _hit64(V, F, o, d, tri.clamp(min=0))
        return [None, torch.where((tri < 0)[:, None], 0.0, torch.stack([t, b1, b2], 1))]
    if kind == "loss":
        x, y = f64(s["img"]), f64(s["target"])
        x.requires_grad_(True)
        col = (((x - y) * y) ** 2).sum(1).mean()
        nx, ny = x.norm(dim=1), y.norm(dim=1)
        live = (nx.detach() > 0) & (ny > 0)
        cos = torch.zeros_like(ny)
        cos[live] = (x[live] * y[live]).sum(1) / (nx[live] * ny[live])
        tone = ((1 - cos) ** 2 - y.var(dim=1, unbiased=False)).mean()
        total = col + 0.5 * tone
        return [torch.autograd.grad(total, x)[0], torch.stack([total, col, tone]).detach()]
    V, F = f64(s["V"]), s["F"].long().to(_dev64())
    i, j, deg = _laplacian64(F, len(V))
    if kind == "edge":
        V.requires_grad_(True)
        n = torch.nn.functional.normalize(_normals64(V, F), dim=1)
        loss = ((1 - (n[i] * n[j]).sum(1)) ** 2).mean()  # both directions of every edge
        return [loss.detach().reshape(1), torch.autograd.grad(loss, V)[0]]
    lam, lr = 10.0, float(np.float32(1e-3))
    b1, b2 = float(np.float32(0.9)), float(np.float32(0.999))
    g = _solve64(i, j, deg, lam, f64(s["g"]))
    m, v = (1 - b1) * g, (1 - b2) * (g * g).max()
    u = V + lam * (deg[:, None] * V - torch.zeros_like(V).index_add(0, i, V[j]))
    u = u - lr * (m / (1 - b1)) / (torch.sqrt(v / (1 - b2)) + 1e-8)
    return [_solve64(i, j, deg, lam, u), m.reshape(-1)]
