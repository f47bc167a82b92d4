"""Timed cases of the framework: the calls of a latent-feature mapping session, from the smallest
optimisation step to the decode of a building-sized keyframe.

`listed()` names the cases, `draw()` gives further ones of the same ranges, `prepare()` makes on
the GPU what a program holds before the call, `run()` is one pass through the public API and
`exact()` the same results in 64 bits from plain PyTorch.  `work()` counts the bytes (each input
read once, each output written once) and the floating-point operations no implementation can do
without.

Inputs are seeded and synthetic: rooms of 6 x 5 x 3 m with 20 boxes, a two-floor building,
targets that are piecewise constant over surface segments plus noise and unit length per row, and
cell masks of the segments (what an automatic mask generator gives on walls and floors).
"""
from __future__ import annotations

import math
import random
from types import SimpleNamespace

import numpy as np
import torch

from paper_2602_12314_gb300 import api

PRECISIONS = {"fp32": api.FP32, "bf16": api.BF16, "fp8": api.FP8}
ROOM = (6.0, 5.0, 3.0)
TILE = 16
LR, BETA1, BETA2, EPS, ADAM_STEP = 0.01, 0.9, 0.999, 1e-8, 20  # mid-optimisation: moments not zero


def listed():
    return [
        # the smallest optimisation step: one view of a toy scene, bound by latency and launches
        dict(name="step_tiny", kind="step", width=64, height=48, gaussians=2000, d=16, M=64, D=512,
             precision="fp32"),
        # one whole iteration on a room keyframe with per-pixel targets
        dict(name="step_room", kind="step", width=640, height=480, gaussians=300_000, d=32, M=256, D=512,
             precision="fp32"),
        # Algorithm 1 on one new keyframe and five of the history with mask-pooled targets: one
        # iteration on queries and dictionary, five on the dictionary alone
        dict(name="keyframe_masks", kind="keyframe", views=6, width=640, height=480, gaussians=300_000, d=32, M=256,
             D=512, precision="fp32"),
        # the dictionary decode with loss and backward for per-pixel targets of a room keyframe
        dict(name="decode_train_room", kind="decode_train", rows=640 * 480, d=32, M=256, D=512, precision="fp32",
             target="fp32", tau=0.0),
        # the same for a building keyframe with the largest dictionary, in BF16
        dict(name="decode_train_building", kind="decode_train", rows=1296 * 968, d=32, M=1024, D=768,
             precision="bf16", target="bf16", tau=0.0),
        # features of a rendered 1200 x 680 view for open-vocabulary queries (no loss, no gradient)
        dict(name="decode_view", kind="decode_fwd", rows=1200 * 680, d=32, M=512, D=768, precision="bf16"),
        # rendering that view's query image: projection, binning, blend
        dict(name="splat_view", kind="splat", width=1200, height=680, gaussians=600_000, d=32),
        # gradient of the queries from an 848 x 480 query-image gradient
        dict(name="splat_grad", kind="splat_grad", width=848, height=480, gaussians=200_000, d=32),
        # gradients of the full mapping objective (geometry, colour, depth, features)
        dict(name="objective_room", kind="objective", width=640, height=480, gaussians=300_000, d=32, M=256, D=512,
             precision="fp32"),
        # the dictionary's streaming K-means update from a keyframe's mask targets ...
        dict(name="kmeans_masks", kind="kmeans", rows=95, D=512, K=256, micro=5),
        # ... and from its per-pixel targets
        dict(name="kmeans_pixels", kind="kmeans", rows=640 * 480, D=512, K=256, micro=5),
        # moving the active local map of a 2M-Gaussian building along the camera's path
        dict(name="map_sync", kind="map", gaussians=2_000_000, d=32, radius=5.0, host=False),
    ]


def _log(rng: random.Random, lo: float, hi: float) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["step", "keyframe", "decode_train", "decode_train", "decode_fwd", "splat", "splat_grad",
                       "objective", "kmeans", "kmeans", "map"])
    d = rng.choice([16, 32, 32, 64])
    dims = dict(d=d, M=32 * _log(rng, 2, 32), D=128 * _log(rng, 1, 8))
    if kind in ("step", "objective"):
        w = _log(rng, 64, 848 if kind == "step" else 640)
        return dict(kind=kind, width=w, height=max(16, int(w * rng.uniform(0.5, 0.8))),
                    gaussians=_log(rng, 2000, 400_000), precision=rng.choice(["fp32", "bf16"]) if kind == "step" else
                    "fp32", **dict(dims, M=32 * _log(rng, 2, 16)))
    if kind == "keyframe":
        w = _log(rng, 160, 848)
        return dict(kind=kind, views=rng.randint(1, 8), width=w, height=int(w * rng.uniform(0.5, 0.8)),
                    gaussians=_log(rng, 20_000, 400_000), precision="fp32", **dims)
    if kind == "decode_train":
        most = min(1296 * 968, 1296 * 968 * 1024 * 768 // (2 * dims["M"] * dims["D"]))
        precision = rng.choice(["fp32", "bf16"])
        tau = rng.choice([0.0, 0.0, 0.1]) if precision == "fp32" else 0.0
        return dict(kind=kind, rows=_log(rng, 90, most), precision=precision, target=rng.choice(["fp32", "bf16"]),
                    tau=tau, **dims)
    if kind == "decode_fwd":
        return dict(kind=kind, rows=_log(rng, 1000, 1_000_000), precision=rng.choice(["fp32", "bf16", "fp8"]), **dims)
    if kind in ("splat", "splat_grad"):
        w = _log(rng, 96, 1296)
        return dict(kind=kind, width=w, height=max(16, int(w * rng.uniform(0.5, 0.8))),
                    gaussians=_log(rng, 5000, 1_000_000), d=d)
    if kind == "kmeans":
        return dict(kind=kind, rows=_log(rng, 40, 400_000), D=128 * _log(rng, 2, 8), K=_log(rng, 64, 2000),
                    micro=rng.choice([5, 5, 8, 13]))
    return dict(kind=kind, gaussians=_log(rng, 50_000, 2_000_000), d=d, radius=round(rng.uniform(2.0, 6.0), 2),
                host=rng.random() < 0.25)


# ---- inputs --------------------------------------------------------------------------------

_CTX = None


def _ctx():
    """The program's one library context."""
    global _CTX
    if _CTX is None:
        _CTX = api.Context()
    return _CTX


def _gen(seed: int):
    return torch.Generator(device="cuda").manual_seed(seed)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda")


def _unit(x):
    return x / x.norm(dim=-1, keepdim=True).clamp_min(1e-12)


def _boxes(rng: np.random.Generator, n: int = 20):
    out = []
    for _ in range(n):
        e = rng.uniform(0.2, 1.0, 3)
        lo = np.array([rng.uniform(0.1, ROOM[0] - e[0] - 0.1), rng.uniform(0.1, ROOM[1] - e[1] - 0.1), 0.0])
        out.append((lo, lo + e))
    return out


def _box_faces(lo, hi, axes):
    """(origin, edge u, edge v, normal axis) of the faces of an axis-aligned box normal to `axes`."""
    faces = []
    for ax in axes:
        for side in (lo, hi):
            u, v = [a for a in range(3) if a != ax]
            o, eu, ev = np.array(lo, float), np.zeros(3), np.zeros(3)
            o[ax], eu[u], ev[v] = side[ax], hi[u] - lo[u], hi[v] - lo[v]
            faces.append((o, eu, ev, ax))
    return faces


def _surface(g, faces, n: int, d: int) -> dict:
    """n Gaussians spread over the faces in proportion to area, flat along the normal, ~1.5 cm."""
    t = lambda a: torch.as_tensor(np.array(a), dtype=torch.float32, device="cuda")  # noqa: E731
    O, U, V = (t([f[k] for f in faces]) for k in range(3))
    ax = torch.as_tensor([f[3] for f in faces], device="cuda")
    area = torch.linalg.cross(U, V).norm(dim=1)
    which = torch.searchsorted(torch.cumsum(area, 0) / area.sum(), torch.rand(n, generator=g, device="cuda"))
    which = which.clamp_max(len(faces) - 1)
    ab = torch.rand(n, 2, generator=g, device="cuda")
    scales = torch.exp(_randn(g, n, 3) * 0.3 + math.log(0.015))
    rows = torch.arange(n, device="cuda")
    scales[rows, ax[which]] *= 0.3
    theta = torch.rand(n, generator=g, device="cuda") * math.pi
    quats = torch.zeros(n, 4, device="cuda")
    quats[:, 0] = torch.cos(theta)
    quats[rows, 1 + ax[which]] = torch.sin(theta)
    return dict(means=(O[which] + ab[:, :1] * U[which] + ab[:, 1:] * V[which]).contiguous(), quats=quats,
                scales=scales, opacities=0.3 + 0.69 * torch.rand(n, generator=g, device="cuda"), f=_randn(g, n, d))


def _camera(rng: np.random.Generator, width: int, height: int, jitter: float = 0.0):
    yaw = rng.uniform(0, 2 * math.pi)
    pos = np.array([ROOM[0] / 2, ROOM[1] / 2, 1.5]) + jitter * rng.uniform(-1.0, 1.0, 3)
    fwd = np.array([math.cos(yaw), math.sin(yaw), 0.0])
    down = np.array([0.0, 0.0, -1.0])
    R = np.stack([np.cross(down, fwd), down, fwd]).astype(np.float32)
    return SimpleNamespace(R=R, t=(-R @ pos).astype(np.float32), fx=525.0 * width / 640.0, fy=525.0 * width / 640.0,
                           cx=width / 2, cy=height / 2, width=width, height=height, z_near=0.2)


def _raycast(cam, boxes):
    """Segment id (boxes, then two halves of every room plane) and camera depth of every pixel."""
    y, x = torch.meshgrid(torch.arange(cam.height, device="cuda", dtype=torch.float64),
                          torch.arange(cam.width, device="cuda", dtype=torch.float64), indexing="ij")
    R = torch.as_tensor(cam.R, dtype=torch.float64, device="cuda")
    dirw = (torch.stack([(x - cam.cx) / cam.fx, (y - cam.cy) / cam.fy, torch.ones_like(x)], -1).reshape(-1, 3)) @ R
    o = -R.T @ torch.as_tensor(cam.t, dtype=torch.float64, device="cuda")
    best = torch.full((dirw.shape[0],), math.inf, dtype=torch.float64, device="cuda")
    label = torch.zeros(dirw.shape[0], dtype=torch.int64, device="cuda")
    for ax in range(3):  # the room seen from inside
        t = torch.where(dirw[:, ax] > 0, ROOM[ax] - o[ax], -o[ax]) / dirw[:, ax]
        u = (ax + 1) % 3
        half = (o[u] + t * dirw[:, u] > ROOM[u] / 2).long()
        hit = (t > 1e-9) & (t < best)
        best = torch.where(hit, t, best)
        label = torch.where(hit, len(boxes) + 4 * ax + 2 * (dirw[:, ax] > 0).long() + half, label)
    for b, (lo, hi) in enumerate(boxes):
        a = (torch.as_tensor(lo, device="cuda") - o) / dirw
        c = (torch.as_tensor(hi, device="cuda") - o) / dirw
        near, far = torch.minimum(a, c).amax(1), torch.maximum(a, c).amin(1)
        hit = (far >= near) & (near > 1e-9) & (near < best)
        best = torch.where(hit, near, best)
        label = torch.where(hit, b, label)
    return label, torch.where(torch.isfinite(best), best, torch.zeros_like(best)).float()


def _targets(g, emb, label):
    """Unit target rows: the segment's embedding plus noise."""
    F = emb[label]
    F += 0.02 * _randn(g, *F.shape)
    F /= F.norm(dim=1, keepdim=True)
    return F


def _dictionary(g, M, d, D):
    K, V = _randn(g, M, d) / math.sqrt(d), _randn(g, M, D) / math.sqrt(d)
    return K, V, V - 0.1 * _unit(_randn(g, M, D)) * (2.0 * torch.rand(M, 1, generator=g, device="cuda"))


def _room(case, g, rng, views: int):
    """The room's Gaussians, boxes and cameras."""
    boxes = _boxes(rng)
    faces = _box_faces(np.zeros(3), np.array(ROOM), range(3))
    for lo, hi in boxes:
        faces += _box_faces(lo, hi, range(3))
    cams = [_camera(rng, case["width"], case["height"], 0.3 if k else 0.0) for k in range(views)]
    return _surface(g, faces, case["gaussians"], case["d"]), boxes, cams


def _masks(g, cam, label, emb, cell=80):
    """CSR pixel lists of the (segment, image cell) pairs, their targets and loss flags."""
    pix = torch.arange(label.numel(), device="cuda")
    ncx = (cam.width + cell - 1) // cell
    key = label * 100_000 + (pix // cam.width // 60) * ncx + (pix % cam.width) // cell
    order = torch.sort(key, stable=True).indices
    uniq, counts = torch.unique_consecutive(key[order], return_counts=True)
    off = torch.zeros(uniq.numel() + 1, dtype=torch.int64, device="cuda")
    off[1:] = torch.cumsum(counts, 0)
    F = _unit(emb[uniq // 100_000] + 0.005 * _randn(g, uniq.numel(), emb.shape[1]))
    valid = (torch.rand(uniq.numel(), generator=g, device="cuda") > 0.1).to(torch.uint8)
    return SimpleNamespace(offsets=off.int(), pixels=order.int(), F=F, valid=valid)


def _moments(g, like, scale):
    """Adam moments of a running optimisation whose gradients have the given scale."""
    return (scale * _randn(g, *like.shape)).contiguous(), torch.full_like(like, scale * scale)


def prepare(case, seed):
    g, rng = _gen(seed), np.random.default_rng(seed)
    kind = case["kind"]
    s = SimpleNamespace(kind=kind, case=case)
    if kind in ("step", "keyframe", "objective"):
        geo, boxes, cams = _room(case, g, rng, case.get("views", 1))
        emb = _unit(_randn(g, len(boxes) + 12, case["D"]))
        K, V, V0 = _dictionary(g, case["M"], case["d"], case["D"])
        scenes = []
        for cam in cams:
            label, depth = _raycast(cam, boxes)
            mask = (torch.rand(label.numel(), generator=g, device="cuda") > 0.05).to(torch.uint8)
            F = _targets(g, emb, label) if kind != "keyframe" else None
            scenes.append(SimpleNamespace(**geo, K=K, V=V, V0=V0, F=F, mask=mask, camera=cam, label=label,
                                          depth=depth))
        adam = api.AdamConfig(lr_f=LR, lr_dict=LR, beta1=BETA1, beta2=BETA2, eps=EPS, step=ADAM_STEP)
        if kind == "objective":
            s.scene = scenes[0]
            seg = torch.rand(len(boxes) + 12, 3, generator=g, device="cuda")
            s.colours = torch.rand(case["gaussians"], 3, generator=g, device="cuda")
            image = seg[scenes[0].label]
            s.image = (image + 0.02 * _randn(g, *image.shape)).clamp(0.0, 1.0)
        elif kind == "step":
            s.step = api.LatentStep(_ctx(), scenes[0], adam_cfg=adam, precision=PRECISIONS[case["precision"]])
            s.mom = s.step.moments
            for name, scale in (("f", 1e-6), ("K", 1e-4), ("V", 1e-5)):
                s.mom[name], s.mom["v" + name] = _moments(g, s.mom[name], scale)
            s.scenes = scenes
        else:
            s.masks = [_masks(g, sc.camera, sc.label, emb) for sc in scenes]
            s.step = api.LatentBatchStep(_ctx(), scenes, adam_cfg=adam, precision=PRECISIONS[case["precision"]],
                                         masks=s.masks)
            geo_, (f, _, _), cam_ = s.step.frames[0]
            s.q = (f, *_moments(g, f, 1e-6))  # every view shares the map's queries and moments
            s.step.frames = [(ge, s.q, ca) for ge, _, ca in s.step.frames]
            s.step.mK, s.step.vK = _moments(g, s.step.K, 1e-4)
            s.step.mV, s.step.vV = _moments(g, s.step.V, 1e-5)
            s.scenes = scenes
    elif kind in ("decode_train", "decode_fwd"):
        n, d, M, D = case["rows"], case["d"], case["M"], case["D"]
        s.Q = _randn(g, n, d)
        s.K, s.V, s.V0 = _dictionary(g, M, d, D)
        if kind == "decode_train":
            emb = _unit(_randn(g, 32, D))
            s.F = torch.empty(n, D, device="cuda", dtype=torch.float32 if case["target"] == "fp32" else torch.bfloat16)
            label = torch.randint(32, ((n + 63) // 64,), generator=g, device="cuda").repeat_interleave(64)[:n]
            for i in range(0, n, 1 << 17):
                s.F[i:i + (1 << 17)] = _targets(g, emb, label[i:i + (1 << 17)])
            s.mask = (torch.rand(n, generator=g, device="cuda") > 0.1).to(torch.uint8)
            s.W = _randn(g, d, D) / math.sqrt(d)
    elif kind in ("splat", "splat_grad"):
        s.geo, _, (s.cam,) = _room(case, g, rng, 1)
        if kind == "splat_grad":
            ge = s.geo
            s.proj = api.project(_ctx(), ge["means"], ge["quats"], ge["scales"], ge["opacities"], s.cam)
            s.bins = api.sort(_ctx(), s.proj, s.cam)
            s.nc = api.render_fwd(_ctx(), s.proj, s.cam, s.bins, ge["f"])[2]
            s.dQ = 1e-4 * _randn(g, case["width"] * case["height"], case["d"])
    elif kind == "kmeans":
        n, D, K = case["rows"], case["D"], case["K"]
        emb = _unit(_randn(g, 32, D))
        label = torch.randint(32, ((n + 15) // 16,), generator=g, device="cuda").repeat_interleave(16)[:n]
        label = label if n > 2000 else torch.randint(32, (n,), generator=g, device="cuda")
        s.F = _targets(g, emb, label)
        s.valid = (torch.rand(n, generator=g, device="cuda") > 0.05).to(torch.uint8)
        # half of the slots are taken: older embeddings and what they summarise
        s.C = _unit(_randn(g, K, D))
        s.C[:K // 2] = _unit(emb[torch.arange(K // 2, device="cuda") % 32] + 0.5 * s.C[:K // 2])
        s.w = torch.zeros(K, device="cuda")
        s.w[:K // 2] = torch.randint(n // 8 + 1, n + 2, (K // 2,), generator=g, device="cuda").float()
        rows = np.flatnonzero(s.valid.cpu().numpy())
        s.init = rng.choice(rows, size=min(case["micro"], rows.size), replace=False).astype(np.int32)
    else:
        faces = [(np.array([0, 0, z]), np.array([20.0, 0, 0]), np.array([0, 15.0, 0]), 2) for z in (0.0, 3.0, 6.0)]
        faces += [(np.array([x, 0, 0]), np.array([0, 15.0, 0]), np.array([0, 0, 6.0]), 0) for x in range(0, 21, 5)]
        faces += [(np.array([0, y, 0]), np.array([20.0, 0, 0]), np.array([0, 0, 6.0]), 1) for y in range(0, 16, 5)]
        # where the Gaussians and the path lie is the building's; what they carry is the seed's
        ge, rng = _surface(_gen(0), faces, case["gaussians"], case["d"]), np.random.default_rng(0)
        ge["f"] = _randn(g, case["gaussians"], case["d"])
        ge["opacities"] = 0.3 + 0.69 * torch.rand(case["gaussians"], generator=g, device="cuda")
        s.map = api.VoxelMap(_ctx(), case["d"], table_log2=24, voxel_size=0.05, capacity=case["gaussians"],
                             host_store=case["host"])
        s.map.insert(ge["means"], ge["quats"], ge["scales"], ge["opacities"], ge["f"])
        a = rng.uniform(0, 2 * math.pi)  # two neighbouring keyframes of the path, visited in turn
        c0 = np.array([rng.uniform(5, 15), rng.uniform(5, 10), 1.5])
        s.path = [c0.tolist(), (c0 + [0.8 * math.cos(a), 0.8 * math.sin(a), 0.0]).tolist()]
        s.at = 0
        s.map.sync(s.path[1], case["radius"])
    return s


class _Local(dict):
    """A map's local rows, which are views of the map's memory: holding them holds the map."""


# ---- the calls -------------------------------------------------------------------------------

def run(s):
    case, kind = s.case, s.kind
    if kind == "step":
        loss = s.step.step()
        return dict(loss=loss, f=s.step.f, K=s.step.K, V=s.step.V, moments=s.step.moments)
    if kind == "keyframe":
        first = s.step.step(1, learn_f=True)
        last = s.step.step(5, learn_f=False)
        st = s.step
        return dict(first=first, last=last, f=s.q[0], m_f=s.q[1], v_f=s.q[2], K=st.K, V=st.V, mK=st.mK, vK=st.vK,
                    mV=st.mV, vV=st.vV)
    if kind == "objective":
        sc = s.scene
        return api.backward_full(_ctx(), sc.means, sc.quats, sc.scales, sc.opacities, s.colours, sc.f, sc.camera,
                                 sc.K, sc.V, sc.V0, sc.F, sc.mask, s.image, sc.depth,
                                 precision=PRECISIONS[case["precision"]])
    if kind == "decode_train":
        prec = PRECISIONS[case["precision"]]
        if case["tau"] > 0:
            return api.decode_loss_bwd_paper(_ctx(), s.Q, s.W, s.V, s.V0, s.F, case["tau"], s.mask, precision=prec)
        return api.decode_loss_bwd(_ctx(), s.Q, s.K, s.V, s.V0, s.F, s.mask, precision=prec)
    if kind == "decode_fwd":
        return api.decode_fwd(_ctx(), s.Q, s.K, s.V, precision=PRECISIONS[case["precision"]])
    if kind == "splat":
        ge = s.geo
        proj = api.project(_ctx(), ge["means"], ge["quats"], ge["scales"], ge["opacities"], s.cam)
        bins = api.sort(_ctx(), proj, s.cam)
        Q, T, nc = api.render_fwd(_ctx(), proj, s.cam, bins, ge["f"])
        return dict(xy=proj.xy, conic_opacity=proj.conic_opacity, depth=proj.depth, rect=proj.rect,
                    tiles=proj.tiles_touched, pairs=bins.num_pairs, ranges=bins.tile_ranges, Q=Q, T=T,
                    n_contrib=nc)
    if kind == "splat_grad":
        return api.render_bwd(_ctx(), s.proj, s.cam, s.bins, s.nc, s.dQ)
    if kind == "kmeans":
        api.stream_kmeans(_ctx(), s.F, s.C, s.w, s.init, valid=s.valid)
        return s.C, s.w
    s.at ^= 1
    local = _Local(s.map.sync(s.path[1 - s.at], case["radius"]))
    local.map = s.map
    return local


def work(case):
    kind, d, D = case["kind"], case.get("d", 0), case.get("D", 0)
    M, N = case.get("M", 0), case.get("gaussians", 0)
    n = case.get("rows", 0) or case.get("width", 0) * case.get("height", 0)
    dic = M * (d + D)
    if kind == "decode_fwd":
        return dict(bytes=4 * (n * d + dic + n * D + 2 * n), flops=2 * n * M * (d + D))
    if kind == "decode_train":
        e = 4 if case["target"] == "fp32" else 2
        return dict(bytes=n * (8 * d + e * D + 1) + 4 * (3 * dic), flops=6 * n * M * (d + D))
    if kind == "kmeans":
        return dict(bytes=4 * n * D + 8 * case["K"] * D,
                    flops=10 * 2 * D * (n * (case["micro"] + 1) + case["K"] * (case["K"] // 2 + case["micro"])))
    if kind == "map":
        local = N * min(1.0, 1.2 * case["radius"] ** 2 / 300.0)
        return dict(bytes=12 * N + 2 * local * (52 + 12 * d), flops=8 * N)
    pairs = 0.4 * N  # about what a room view sees of its map
    splat = dict(bytes=N * 92 + pairs * 4 * d + n * (4 * d + 8), flops=pairs * 256 * (2 * d + 12))
    if kind == "splat":
        return splat
    if kind == "splat_grad":
        return dict(bytes=pairs * 28 + 4 * n * (d + 1) + 4 * N * d, flops=pairs * 256 * (2 * d + 12))
    dec = dict(bytes=n * (8 * d + 4 * D + 1) + 12 * dic, flops=6 * n * M * (d + D))
    if kind == "objective":
        return dict(bytes=splat["bytes"] + dec["bytes"] + n * (8 * d + 48) + N * (8 * d + 120),
                    flops=3 * splat["flops"] + dec["flops"] + 700 * n)
    adam = 28 * (N * d + dic)
    if kind == "step":
        return dict(bytes=splat["bytes"] + dec["bytes"] + 4 * n * d + adam, flops=2 * splat["flops"] + dec["flops"])
    v = case["views"]
    masks = 100 * v
    return dict(bytes=v * (2 * splat["bytes"] + 4 * n * (d + 1)) + masks * 6 * 4 * (D + d) + adam + 5 * 28 * dic,
                flops=v * 3 * splat["flops"] + 6 * 6 * masks * M * (d + D))


# ---- the same results in 64 bits -------------------------------------------------------------

def _project64(means, quats, scales, cam):
    """Screen means, conics, 2D covariance diagonal, camera depth (all differentiable)."""
    f32 = lambda x: float(np.float32(x))  # noqa: E731
    R = torch.as_tensor(cam.R, dtype=torch.float64, device="cuda")
    p = means @ R.T + torch.as_tensor(cam.t, dtype=torch.float64, device="cuda")
    x, y, z = p.unbind(1)
    w, a, b, c = (quats / quats.norm(dim=1, keepdim=True)).unbind(1)
    rot = torch.stack([1 - 2 * (b * b + c * c), 2 * (a * b - w * c), 2 * (a * c + w * b),
                       2 * (a * b + w * c), 1 - 2 * (a * a + c * c), 2 * (b * c - w * a),
                       2 * (a * c - w * b), 2 * (b * c + w * a), 1 - 2 * (a * a + b * b)], 1).reshape(-1, 3, 3)
    fx, fy, o = f32(cam.fx), f32(cam.fy), torch.zeros_like(z)
    J = torch.stack([fx / z, o, -fx * x / (z * z), o, fy / z, -fy * y / (z * z)], 1).reshape(-1, 2, 3)
    B = (J @ R) @ (rot * scales[:, None, :])
    S = B @ B.transpose(1, 2)
    ca, cb, cc = S[:, 0, 0] + 0.3, S[:, 0, 1], S[:, 1, 1] + 0.3
    det = ca * cc - cb * cb
    uv = torch.stack([fx * x / z + f32(cam.cx), fy * y / z + f32(cam.cy)], 1)
    return uv, torch.stack([cc / det, -cb / det, ca / det], 1), torch.stack([ca, cc], 1), z


def _tile_lists(means32, opac, uv, cov, cam):
    """Front-to-back Gaussian ids of every 16 x 16 tile (a few that reach no pixel among them)."""
    x, y, z = means32.unbind(1)
    r, t2 = [float(v) for v in np.asarray(cam.R, np.float32)[2]], float(np.float32(cam.t[2]))
    key = ((r[0] * x + r[1] * y) + r[2] * z) + t2  # binary32, every operation rounded
    ext = torch.sqrt((2 * torch.log(255 * opac)).clamp_min(0)[:, None] * cov) + 0.01
    tx, ty = (cam.width + TILE - 1) // TILE, (cam.height + TILE - 1) // TILE
    top = torch.tensor([tx, ty], device="cuda", dtype=torch.float64)
    lo = torch.floor((uv - ext) / TILE).clamp_min(0).minimum(top)
    hi = (torch.floor((uv + ext) / TILE) + 1).clamp_min(0).minimum(top)
    seen = (key > cam.z_near) & (opac >= 1 / 255)
    size = torch.where(seen[:, None], torch.nan_to_num(hi - lo).clamp_min(0), torch.zeros_like(lo)).long()
    lo = torch.nan_to_num(lo).long()
    count = size[:, 0] * size[:, 1]
    ids = torch.repeat_interleave(torch.arange(count.numel(), device="cuda"), count)
    k = torch.arange(ids.numel(), device="cuda") - (torch.cumsum(count, 0) - count)[ids]
    tile = (lo[ids, 1] + k // size[ids, 0].clamp_min(1)) * tx + lo[ids, 0] + k % size[ids, 0].clamp_min(1)
    order = torch.sort(key[ids], stable=True).indices
    order = order[torch.sort(tile[order], stable=True).indices]
    ends = torch.cumsum(torch.bincount(tile, minlength=tx * ty), 0).tolist()
    ids = ids[order]
    return [ids[a:b] for a, b in zip([0] + ends[:-1], ends)]


def _blend64(ids, tile, uv, conic, opac, cam):
    """Pixels of the tile and their blend weights (pixels x list), and the transmittance left."""
    tx = (cam.width + TILE - 1) // TILE
    y, x = torch.meshgrid(torch.arange(tile // tx * TILE, min(tile // tx * TILE + TILE, cam.height), device="cuda"),
                          torch.arange(tile % tx * TILE, min(tile % tx * TILE + TILE, cam.width), device="cuda"),
                          indexing="ij")
    x, y = x.reshape(-1), y.reshape(-1)
    u, q = uv[ids], conic[ids]
    dx, dy = u[None, :, 0] - x[:, None], u[None, :, 1] - y[:, None]
    power = -0.5 * (q[:, 0] * dx * dx + q[:, 2] * dy * dy) - q[:, 1] * dx * dy
    alpha = (opac[ids] * torch.exp(power)).clamp_max(0.99)
    alpha = alpha * ((power <= 0) & (alpha >= 1 / 255)).detach()
    after = torch.cumprod(1 - alpha, 1)
    before = torch.cat([torch.ones_like(after[:, :1]), after[:, :-1]], 1)
    keep = (after >= 1e-4).detach()
    left = torch.where(keep, after, torch.ones_like(after)).amin(1) if ids.numel() else torch.ones_like(x).double()
    return y * cam.width + x, alpha * before * keep, left


class _View64:
    """A camera's view of a fixed map in 64 bits: render and its adjoint."""

    def __init__(self, geo, cam):
        self.cam = cam
        d = lambda k: geo[k].double()  # noqa: E731
        self.uv, self.conic, cov, self.z = _project64(d("means"), d("quats"), d("scales"), cam)
        self.opac = d("opacities")
        self.lists = _tile_lists(geo["means"], self.opac, self.uv, cov, cam)

    def tiles(self):
        for t, ids in enumerate(self.lists):
            yield ids, *_blend64(ids, t, self.uv, self.conic, self.opac, self.cam)

    def render(self, f):
        n = self.cam.width * self.cam.height
        Q, T = torch.zeros(n, f.shape[1], dtype=torch.float64, device="cuda"), torch.ones(n, dtype=torch.float64,
                                                                                           device="cuda")
        for ids, pix, w, left in self.tiles():
            if ids.numel():
                Q[pix], T[pix] = w @ f[ids], left
        return Q, T

    def adjoint(self, dQ, df):
        for ids, pix, w, _ in self.tiles():
            if ids.numel():
                df.index_add_(0, ids, w.T @ dQ[pix])


def _decode64(Q, K, V, V0, F, mask, tau=0.0, need_dQ=True):
    """Loss parts and gradients of the feature objective (K is the projection W when tau > 0)."""
    n, d = Q.shape
    cfg = api.LossConfig()
    K, V = (x.double().clone().requires_grad_() for x in (K, V))
    nv = int(mask.sum())
    dQ = torch.zeros(n, d, dtype=torch.float64, device="cuda") if need_dQ else None
    cos_sum, l2_sum = 0.0, 0.0
    for i in range(0, n, 1 << 16):
        r = slice(i, i + (1 << 16))
        q = Q[r].double().detach().requires_grad_(need_dQ)
        keys = V / V.norm(dim=1, keepdim=True) if tau > 0 else K
        x = q @ K if tau > 0 else q
        S = (x / x.norm(dim=1, keepdim=True)) @ keys.T / tau if tau > 0 else q @ keys.T / math.sqrt(d)
        Fh, f, m = torch.softmax(S, 1) @ V, F[r].double(), mask[r].double()
        cos = (Fh * f).sum(1) / (Fh.norm(dim=1) * f.norm(dim=1)).clamp_min(1e-8)
        c, e = (m * (1 - cos)).sum(), (m * (Fh - f).square().sum(1)).sum()
        loss = cfg.lambda_f * (cfg.lambda_cos * c / max(nv, 1) + cfg.lambda_2 * e / (max(nv, 1) * V.shape[1]))
        loss.backward()
        cos_sum, l2_sum = cos_sum + float(c.detach()), l2_sum + float(e.detach())
        if need_dQ:
            dQ[r] = q.grad
    tr = ((V - V0.double()).norm(dim=1) - float(np.float32(cfg.delta))).clamp_min(0).sum()
    (float(np.float32(cfg.lambda_f * cfg.lambda_D)) * tr).backward()
    c, e, tr = cos_sum / max(nv, 1), l2_sum / (max(nv, 1) * V.shape[1]), float(tr.detach())
    total = cfg.lambda_f * (cfg.lambda_cos * c + cfg.lambda_2 * e + cfg.lambda_D * tr)
    return [c, e, tr, total, float(nv)], dQ, K.grad, V.grad


def _adam64(p, g, m, v, step):
    m.mul_(BETA1).add_((1 - BETA1) * g)
    v.mul_(BETA2).add_((1 - BETA2) * g * g)
    p.sub_(LR * (m / (1 - BETA1 ** step)) / ((v / (1 - BETA2 ** step)).sqrt() + EPS))


def _pool64(Q, ms):
    """Mean rows of the masks, and the adjoint of that mean."""
    off = ms.offsets.long()
    owner = torch.repeat_interleave(torch.arange(off.numel() - 1, device="cuda"), off[1:] - off[:-1])
    count = (off[1:] - off[:-1]).double()[:, None]
    pix = ms.pixels.long()
    pooled = torch.zeros(off.numel() - 1, Q.shape[1], dtype=torch.float64, device="cuda")
    pooled.index_add_(0, owner, Q[pix])
    return pooled / count, lambda dQm: torch.zeros_like(Q).index_add_(0, pix, (dQm / count)[owner])


def _exact_steps(s, masks, iterations):
    """f, K, V and their moments after the iterations (True: all three, False: K and V)."""
    sc = s.scenes[0]
    geo = dict(means=sc.means, quats=sc.quats, scales=sc.scales, opacities=sc.opacities)
    views = [_View64(geo, x.camera) for x in s.scenes]
    st = s.step
    if masks is None:
        first = [st.f, st.K, st.V, *(s.mom[k] for k in ("f", "vf", "K", "vK", "V", "vV"))]
    else:
        first = [s.q[0], st.K, st.V, s.q[1], s.q[2], st.mK, st.vK, st.mV, st.vV]
    f, K, V, mf, vf, mK, vK, mV, vV = (x.double().clone() for x in first)
    F, flags, V0 = st.F, st.mask, st.V0
    losses, rendered = [], None
    for i, learn_f in enumerate(iterations):
        if rendered is None or learn_f or iterations[i - 1]:
            rendered = [v.render(f)[0] for v in views]
        pools = [_pool64(q, m) for q, m in zip(rendered, masks)] if masks else None
        rows = torch.cat([p[0] for p in pools]) if masks else rendered[0]
        parts, dQ, dK, dV = _decode64(rows, K, V, V0, F, flags, need_dQ=learn_f)
        losses.append(dict(zip(("cos", "l2", "tr", "total", "n_valid"), parts)))
        if learn_f:
            df = torch.zeros_like(f)
            for k, v in enumerate(views):
                if masks:
                    cut = sum(p[0].shape[0] for p in pools[:k])
                    v.adjoint(pools[k][1](dQ[cut:cut + pools[k][0].shape[0]]), df)
                else:
                    v.adjoint(dQ, df)
            _adam64(f, df, mf, vf, ADAM_STEP + i)
        _adam64(K, dK, mK, vK, ADAM_STEP + i)
        _adam64(V, dV, mV, vV, ADAM_STEP + i)
    return losses, f, K, V, mf, vf, mK, vK, mV, vV


def _exact_objective(s):
    """Gradients of the full mapping objective by automatic differentiation."""
    sc, cam = s.scene, s.scene.camera
    names = ("means", "quats", "scales", "opacities", "f")
    p = {k: getattr(sc, k).double().requires_grad_() for k in names}
    p["colours"] = s.colours.double().requires_grad_()
    uv, conic, cov, z = _project64(p["means"], p["quats"], p["scales"], cam)
    with torch.no_grad():
        lists = _tile_lists(sc.means, p["opacities"], uv, cov, cam)
    screen = [t.detach().requires_grad_() for t in (uv, conic, p["opacities"], p["f"], p["colours"], z)]
    uv_, conic_, op_, f_, c_, z_ = screen
    n, d = cam.width * cam.height, sc.f.shape[1]
    image = torch.zeros(n, d + 4, dtype=torch.float64, device="cuda")
    channels = torch.cat([f_, c_, z_[:, None]], 1)
    with torch.no_grad():
        for t, ids in enumerate(lists):
            if ids.numel():
                pix, w, _ = _blend64(ids, t, uv_, conic_, op_, cam)
                image[pix] = w @ channels[ids]
    parts, dQ, dK, dV = _decode64(image[:, :d], sc.K, sc.V, sc.V0, sc.F, sc.mask)
    C, Z = image[:, d:d + 3].clone().requires_grad_(), image[:, d + 3].clone().requires_grad_()
    y = s.image.double()
    win = torch.exp(-(torch.arange(11, dtype=torch.float64, device="cuda") - 5) ** 2 / 4.5)
    win = (win / win.sum()).float().double()

    def blur(t):
        t = t.T.reshape(3, 1, cam.height, cam.width)
        t = torch.nn.functional.pad(t, (5, 5, 5, 5))
        t = sum(win[k] * t[..., k:k + cam.width] for k in range(11))
        return sum(win[k] * t[:, :, k:k + cam.height] for k in range(11))

    mx, my = blur(C), blur(y)
    sxx, syy, sxy = blur(C * C) - mx * mx, blur(y * y) - my * my, blur(C * y) - mx * my
    ssim = ((2 * mx * my + 1e-4) * (2 * sxy + 9e-4) / ((mx * mx + my * my + 1e-4) * (sxx + syy + 9e-4))).mean()
    seen = sc.depth > 0
    l1, ld = (C - y).abs().mean(), ((Z - sc.depth.double()).abs() * seen).sum() / seen.sum().clamp_min(1)
    (0.2 * l1 + 0.8 * (1 - ssim) + 0.1 * ld).backward()
    G = torch.cat([dQ, C.grad, Z.grad[:, None]], 1)
    grads = [torch.zeros_like(t) for t in screen]
    for t, ids in enumerate(lists):  # tile by tile, over copies of the tile's own rows
        if ids.numel():
            own = [x.detach()[ids].requires_grad_() for x in screen]
            pix, w, _ = _blend64(torch.arange(ids.numel(), device="cuda"), t, own[0], own[1], own[2], cam)
            out = w @ torch.cat([own[3], own[4], own[5][:, None]], 1)
            for acc, part in zip(grads, torch.autograd.grad(out, own, G[pix])):
                acc.index_add_(0, ids, part)
    torch.autograd.backward([uv, conic, z], [torch.nan_to_num(grads[0]), grads[1], grads[5]])
    l1, ls, ld = float(l1.detach()), 1 - float(ssim.detach()), float(ld.detach())
    parts += [l1, ls, ld, float(seen.sum()), 0.2 * l1 + 0.8 * ls + 0.1 * ld + parts[3]]
    return dict(means=p["means"].grad, quats=p["quats"].grad, scales=p["scales"].grad, opacities=grads[2],
                colours=grads[4], f=grads[3], K=dK, V=dV,
                parts=torch.tensor(parts, dtype=torch.float64, device="cuda"))


def _lloyd64(X, w, C, W, active, iterations):
    """Weighted Lloyd iterations in place; an active centre without points keeps its place."""
    idx = torch.nonzero(active)[:, 0]
    for _ in range(iterations):
        c = C[idx]
        sums, tot = torch.zeros_like(c), torch.zeros(idx.numel(), dtype=torch.float64, device="cuda")
        for i in range(0, X.shape[0], 1 << 16):
            x, xw = X[i:i + (1 << 16)].double(), w[i:i + (1 << 16)]
            a = (c.square().sum(1) - 2 * x @ c.T).argmin(1)
            sums.index_add_(0, a, xw[:, None] * x)
            tot.index_add_(0, a, xw)
        C[idx] = torch.where(tot[:, None] > 0, sums / tot.clamp_min(1e-300)[:, None], c)
        W[idx] = tot


def _exact_kmeans(s):
    X = s.F[s.valid.bool()]
    mC = s.F[torch.as_tensor(s.init, device="cuda").long()].double()
    k = mC.shape[0]
    mW, every = torch.zeros(k, dtype=torch.float64, device="cuda"), torch.ones(k, dtype=torch.bool, device="cuda")
    _lloyd64(X, torch.ones(X.shape[0], dtype=torch.float64, device="cuda"), mC, mW, every, 10)
    C, W = s.C.double().clone(), s.w.double().clone()
    live, used, empty = torch.nonzero(mW > 0)[:, 0], torch.nonzero(W > 0)[:, 0], torch.nonzero(W <= 0)[:, 0]
    P, pw = torch.cat([C[used], mC[live]]), torch.cat([W[used], mW[live]])
    order = live[torch.sort(mW[live], descending=True, stable=True).indices][:empty.numel()]
    C[empty[:order.numel()]] = mC[order]
    active = W > 0
    active[empty[:order.numel()]] = True
    _lloyd64(P, pw, C, W, active, 10)
    return C, W


def exact(case, seed):
    kind = case["kind"]
    if kind == "map":
        return None  # rows are moved, not computed
    if kind == "keyframe" and case["views"] * case["width"] * case["height"] > 2_500_000:
        return None
    s = prepare(case, seed)
    if kind == "step":
        losses, f, K, V, mf, vf, mK, vK, mV, vV = _exact_steps(s, None, [True])
        return dict(loss=losses[0], f=f, K=K, V=V, moments=dict(f=mf, vf=vf, K=mK, vK=vK, V=mV, vV=vV))
    if kind == "keyframe":
        losses, f, K, V, mf, vf, mK, vK, mV, vV = _exact_steps(s, s.masks, [True] + 5 * [False])
        return dict(first=losses[0], last=losses[-1], f=f, m_f=mf, v_f=vf, K=K, V=V, mK=mK, vK=vK, mV=mV, vV=vV)
    if kind == "objective":
        return _exact_objective(s)
    if kind == "decode_train":
        parts, dQ, dK, dV = _decode64(s.Q, s.W if case["tau"] > 0 else s.K, s.V, s.V0, s.F, s.mask, case["tau"])
        return torch.tensor(parts, dtype=torch.float64, device="cuda"), dQ, dK, dV
    if kind == "decode_fwd":
        Fh = torch.empty(case["rows"], case["D"], dtype=torch.float64, device="cuda")
        stats = torch.empty(case["rows"], 2, dtype=torch.float64, device="cuda")
        K, V = s.K.double(), s.V.double()
        for i in range(0, case["rows"], 1 << 16):
            S = s.Q[i:i + (1 << 16)].double() @ K.T / math.sqrt(case["d"])
            top = S.amax(1, keepdim=True)
            e = torch.exp(S - top)
            Fh[i:i + (1 << 16)] = (e @ V) / e.sum(1, keepdim=True)
            stats[i:i + (1 << 16)] = torch.cat([top, e.sum(1, keepdim=True)], 1)
        return Fh, stats
    if kind == "kmeans":
        return _exact_kmeans(s)
    view = _View64(s.geo, s.cam)
    if kind == "splat":
        Q, T = view.render(s.geo["f"].double())
        # the screen-space rows of Gaussians out of view are zero and the depth is a binary32 key
        return dict(xy=None, conic_opacity=None, depth=None, rect=None, tiles=None, pairs=None, ranges=None, Q=Q, T=T,
                    n_contrib=None)
    df = torch.zeros(case["gaussians"], case["d"], dtype=torch.float64, device="cuda")
    view.adjoint(s.dQ.double(), df)
    return df
