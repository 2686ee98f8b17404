"""Workloads of the BG-Triangle rasterizer for performance measurements.

Every case goes through the package's public entry points as a user's program
calls them: training steps (forward, loss gradient, backward) of one view and
of batches, frames rendered for viewing, the photometric loss on its own, and
the densification work between training iterations. Scenes follow the
configurations of scenes.py (split octahedron, icosphere, sphere with three
ellipsoids, room with cubes and spheres), generated here array-wise so that
inputs of a new seed are quick: same meshes, sizes and distributions.

  listed()             the fixed cases
  draw(rng)            one more case of the same ranges
  prepare(case, seed)  inputs and handles on the GPU
  run(state)           one pass, its outputs
  work(case)           bytes and operations one pass cannot do without
  exact(case, seed)    the outputs in FP64, in plain torch
"""
import math

import numpy as np
import torch

from paper_2503_13961_gb300 import render as R
from paper_2503_13961_gb300 import scenes

TESS = 8                       # lattice level of the tessellation (the renderer's default)
PARAMS = ("ctrl", "color", "opacity", "r_b", "log_scale", "quat", "sh")
MIX = (256, 512, 800, 1024)    # view sizes of the batched training workload
MAX_PIXELS = 33_000_000        # pixels of the largest batch


def _render(kind, scene, detail, views, width, height, **over):
    """A rendering case; width = 0: views of the sizes of MIX, drawn by the seed."""
    case = {"kind": kind, "scene": scene, "detail": detail, "degree": 2, "views": views, "width": width,
            "height": height, "r_b": 1e-2, "attr_res": 1, "sh": 0, "loss": "eq9", "autograd": False, "graph": False}
    case.update(over)
    return case


def listed():
    return [
        # the first thing a new user runs: 16 patches, one 64 x 64 view, one training step (launches, latency)
        dict(_render("step", "octa", 1, 1, 64, 64, autograd=True), name="first step 64"),
        # a small ragged photograph, 2,000 patches: one iteration of a PyTorch training loop
        dict(_render("step", "ico", 10, 1, 237, 181, autograd=True), name="step 237x181"),
        # the paper's training iteration at NeRF-Synthetic resolution: one 800^2 view, 20,000 patches, Eq. 9
        dict(_render("step", "blobs", 20, 1, 800, 800, autograd=True), name="step 800"),
        # rotation / scaling maps of leg 3 and SH colour (the paper's full representation), a few views a step
        dict(_render("step", "blobs", 20, 4, 512, 512, attr_res=3, sh=3), name="step maps sh 4x512"),
        # a batch at the paper's finer boundary scale, captured in CUDA graphs, fitting an L1 target
        dict(_render("step", "blobs", 20, 12, 0, 0, r_b=1e-3, loss="l1", graph=True), name="step fine 12 mixed"),
        # the batched training step: 64 views of mixed size in one call
        dict(_render("step", "blobs", 20, 64, 0, 0, loss="l1", graph=True), name="step 64 mixed"),
        # a large indoor scene (100,000 degree-3 patches, dense tiles) under eight 1600 x 1200 views
        dict(_render("step", "room", 40, 8, 1600, 1200, degree=3, loss="l1"), name="step room 8x1600"),
        # one frame of an interactive viewer: an object at 1024^2, the room at 1600 x 1200
        dict(_render("frame", "blobs", 20, 1, 1024, 1024), name="frame 1024"),
        dict(_render("frame", "room", 40, 1, 1600, 1200, degree=3), name="frame room 1600"),
        # Eq. 9 and its image gradient for a batch of views rendered elsewhere
        {"kind": "loss", "views": 64, "width": 0, "height": 0, "lam": 0.2, "name": "loss 64 mixed"},
        # densification between iterations: measures and flags of every primitive, and a quarter of them split
        {"kind": "densify", "prims": 100_000, "degree": 3, "attr_res": 3, "sh": 1, "name": "densify 100k"},
        # the tracking of a period's views: visibility measures, edge magnitudes and their back-projection
        dict(_render("track", "blobs", 20, 64, 0, 0), name="track 64 mixed"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: sizes, counts and options over the whole range of the listed ones."""
    kind = rng.choice(("step", "step", "step", "step", "frame", "frame", "loss", "densify", "track"))
    if kind == "densify":
        return {"kind": kind, "prims": _log_int(rng, 500, 100_000), "degree": rng.randint(1, 4),
                "attr_res": rng.choice((1, 3)), "sh": rng.randint(0, 3)}
    width, height = _log_int(rng, 64, 1600), _log_int(rng, 64, 1200)
    room = kind in ("step", "frame") and rng.random() < 0.25
    most = min(64, max(1, (15_000_000 if room else MAX_PIXELS) // (width * height)))
    views = 1 if kind == "frame" or rng.random() < 0.4 else _log_int(rng, 1, most)
    if not room and kind != "frame" and rng.random() < 0.2:
        width = height = 0
        views = _log_int(rng, 2, 64)
    if kind == "loss":
        return {"kind": kind, "views": views, "width": width, "height": height, "lam": rng.choice((0.2, 0.2, 0.1))}
    if room:
        scene, detail, degree = "room", rng.randint(10, 40), 3
    else:
        scene, detail, degree = rng.choice(("ico", "blobs")), rng.randint(4, 20), rng.choice((1, 2, 2, 2, 3, 4))
    over = {"degree": degree, "r_b": rng.choice((1e-2, 1e-2, 1e-3))}
    if kind == "step":
        over.update(attr_res=rng.choice((1, 1, 3)), sh=rng.choice((0, 0, 1, 3)), loss=rng.choice(("eq9", "l1")))
        over.update(autograd=over["loss"] == "eq9" and rng.random() < 0.5)
        over.update(graph=not over["autograd"] and rng.random() < 0.4)
    return _render(kind, scene, detail, views, width, height, **over)


# ---------------------------------------------------------------------------
# scenes
# ---------------------------------------------------------------------------

def _ncp(n):
    return (n + 1) * (n + 2) // 2


def _orders(n):
    """(i, j, k) of the control points in the library's order."""
    return np.array([(i, j, n - i - j) for i in range(n, -1, -1) for j in range(n - i, -1, -1)], np.float64)


def _lattice(a, b, c, f):
    """f^2 flat triangles of the lattice over the triangles (a, b, c), each [T, 3]."""
    up = [((i, j), (i + 1, j), (i, j + 1)) for i in range(f) for j in range(f - i)]
    down = [((i + 1, j), (i + 1, j + 1), (i, j + 1)) for i in range(f) for j in range(f - 1 - i)]
    ij = np.array(up + down, np.float64)[None, ..., None] / f
    return (a[:, None, None] + (b - a)[:, None, None] * ij[..., 0, :]
            + (c - a)[:, None, None] * ij[..., 1, :]).reshape(-1, 3, 3)


def _ico(f):
    phi = (1 + 5 ** 0.5) / 2
    v = np.array([[-1, phi, 0], [1, phi, 0], [-1, -phi, 0], [1, -phi, 0], [0, -1, phi], [0, 1, phi], [0, -1, -phi],
                  [0, 1, -phi], [phi, 0, -1], [phi, 0, 1], [-phi, 0, -1], [-phi, 0, 1]])
    faces = np.array([(0, 11, 5), (0, 5, 1), (0, 1, 7), (0, 7, 10), (0, 10, 11), (1, 5, 9), (5, 11, 4), (11, 10, 2),
                      (10, 7, 6), (7, 1, 8), (3, 9, 4), (3, 4, 2), (3, 2, 6), (3, 6, 8), (3, 8, 9), (4, 9, 5),
                      (2, 4, 11), (6, 2, 10), (8, 6, 7), (9, 8, 1)])
    t = _lattice(*(v[faces[:, k]] for k in range(3)), f)
    return t / np.linalg.norm(t, axis=-1, keepdims=True)


def _latlong(segments, bands):
    th = np.pi * (np.arange(bands + 1) + 1) / (bands + 2)
    ph = 2 * np.pi * (np.arange(segments + 1) % segments) / segments
    p = np.stack([np.sin(th)[:, None] * np.cos(ph), np.sin(th)[:, None] * np.sin(ph),
                  np.cos(th)[:, None] + 0 * ph], -1)
    a, b, c, d = p[:-1, :-1], p[:-1, 1:], p[1:, :-1], p[1:, 1:]
    return np.stack([np.stack([a, c, b], -2), np.stack([b, c, d], -2)], 2).reshape(-1, 3, 3)


def _box(n):
    """The faces of [-1, 1]^3 as n x n grids."""
    s = np.linspace(-1, 1, n + 1)
    u, v = np.meshgrid(s, s, indexing="ij")
    out = []
    for ax in range(3):
        for sign in (-1.0, 1.0):
            p = np.empty(u.shape + (3,))
            p[..., ax], p[..., (ax + 1) % 3], p[..., (ax + 2) % 3] = sign, u, v
            a, b, c, d = p[:-1, :-1], p[1:, :-1], p[:-1, 1:], p[1:, 1:]
            out.append(np.stack([np.stack([a, b, c], -2), np.stack([b, d, c], -2)], 2).reshape(-1, 3, 3))
    return np.concatenate(out)


def _mesh(case, rng):
    """(triangles [T, 3, 3], centre [T, 3], axes [T, 3]; axes 0: a flat object, object centres)."""
    d = case["detail"]
    parts, centres = [], []

    def add(unit, centre, axes, curved):
        t = unit * axes + centre
        parts.append((t, np.broadcast_to(centre, (len(t), 3)), np.broadcast_to(axes * curved, (len(t), 3))))

    if case["scene"] == "octa":
        add(np.array(scenes.octahedron16_tris()), np.zeros(3), np.ones(3), 1)
    elif case["scene"] in ("ico", "blobs"):
        add(_ico(d), np.zeros(3), np.ones(3), 1)
        if case["scene"] == "blobs":
            unit = _latlong(2 * d, max(2, 5 * d // 2))
            for _ in range(3):
                axes = rng.uniform(0.3, 0.8, 3)
                add(unit, rng.uniform(-1.5, 1.5, 3), axes, 1)
    else:
        add(_box(d), np.zeros(3), np.full(3, 5.0), 0)
        cube, ball = _box(4), _latlong(22, 14)
        for unit, curved, lo, hi in ((cube, 0, 0.15, 0.5), (ball, 1, 0.2, 0.6)):
            for _ in range(round(2.5 * d)):
                centres.append(rng.uniform(-4, 4, 3))
                add(unit, centres[-1], np.full(3, rng.uniform(lo, hi)), curved)
    return tuple(np.concatenate([p[k] for p in parts]) for k in range(3)) + (centres,)


def _scene(case, rng):
    """Scene dict of scenes.py for the case, and the centres of its objects."""
    n = case["degree"]
    tris, centre, axes, centres = _mesh(case, rng)
    ijk = _orders(n)
    p = np.einsum("ac,tcd->tad", ijk / n, tris)
    corner = ijk.max(1) == n
    curved = axes[:, :1, None] > 0
    safe = np.where(axes > 0, axes, 1.0)[:, None]
    x = (p - centre[:, None]) / safe
    on = centre[:, None] + safe * x / np.maximum(np.linalg.norm(x, axis=-1, keepdims=True), 1e-9)
    p = np.where(curved & ~corner[None, :, None], on, p)
    radial = (p - centre[:, None])
    radial /= np.maximum(np.linalg.norm(radial, axis=-1, keepdims=True), 1e-9)
    flat = np.cross(tris[:, 1] - tris[:, 0], tris[:, 2] - tris[:, 0])
    flat /= np.linalg.norm(flat, axis=-1, keepdims=True)
    # one draw per point, shared by the patches that share it (neighbours stay joined)
    key = np.rint(p.reshape(-1, 3) * 2e4).astype(np.int64)
    _, inv = np.unique((key[:, 0] * 2_000_003 + key[:, 1]) * 2_000_003 + key[:, 2], return_inverse=True)
    noise = {"octa": 0.05, "ico": 0.03, "blobs": 0.02, "room": 0.01}[case["scene"]]
    push = rng.normal(0, noise, int(inv.max()) + 1)[inv.reshape(-1)].reshape(p.shape[:2]) * ~corner
    ctrl = p + push[..., None] * np.where(curved, radial, flat[:, None])
    M = len(ctrl)
    dist, width = {"octa": (4.0, 64), "room": (5.0, 1600)}.get(case["scene"], (4.0, 800))
    scale = 0.7 * dist / (width / 2 / math.tan(math.radians(30)))  # 0.7 px at the reference distance
    sc = {"degree": n, "ctrl": ctrl, "color": np.repeat(rng.uniform(0, 1, (M, 1, 3)), _ncp(n), 1),
          "opacity": rng.beta(5, 1, M) if case["scene"] == "room" else rng.uniform(0.5, 1, M),
          "r_b": np.full(M, case["r_b"]), "bg": np.zeros(3),
          # scales and rotations as training leaves them: near the initial ones, no longer isotropic
          "log_scale": math.log(scale) + rng.normal(0, 0.3, (M, 3)),
          "quat": np.array([1.0, 0, 0, 0]) + rng.normal(0, 0.3, (M, 4))}
    if case["attr_res"] > 1:
        sc = scenes.with_attribute_maps(sc, case["attr_res"], seed=int(rng.integers(1 << 30)))
    if case["sh"] > 0:
        sc = scenes.with_sh(sc, case["sh"], seed=int(rng.integers(1 << 30)))
    return sc, centres


def _sizes(case, rng):
    if case["width"]:
        return [(case["width"], case["height"])] * case["views"]
    # mixed sizes whose total does not depend on the seed
    some = [MIX[k % len(MIX)] for k in range(case["views"])]
    return [(int(s), int(s)) for s in rng.permutation(some)]


def _cameras(case, rng, centres):
    sizes = _sizes(case, rng)
    if case["scene"] == "octa":
        return [scenes.look_at_camera((4, rng.uniform(-0.5, 0.5), rng.uniform(-0.5, 0.5)), (0, 0, 0), w, h)
                for w, h in sizes]
    if case["scene"] != "room":
        return scenes.make_views(rng, sizes, 3.5, 5.0)
    cams = []
    for w, h in sizes:
        while True:  # standing in the room, not inside an object
            eye = rng.uniform(-3, 3, 3)
            if min(np.linalg.norm(eye - c) for c in centres) > 1.2:
                break
        cams.append(scenes.look_at_camera(eye, centres[rng.integers(len(centres))], w, h))
    return cams


def _pixels(case):
    if case["width"]:
        return case["views"] * case["width"] * case["height"]
    return sum(MIX[k % len(MIX)] ** 2 for k in range(case["views"]))


def _photos(sizes, seed):
    """Packed images in [0, 1] as a renderer sees them (flat areas, edges, texture) and noisy targets."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    out = []
    for w, h in sizes:
        cells = torch.rand((1, 3, h // 40 + 2, w // 40 + 2), device="cuda", generator=gen)
        flat = torch.nn.functional.interpolate(cells, size=(h, w), mode="nearest")[0].permute(1, 2, 0)
        speck = torch.rand((h, w, 1), device="cuda", generator=gen) < 0.3
        out.append((flat + 0.02 * torch.randn((h, w, 3), device="cuda", generator=gen) * speck).reshape(-1, 3))
    img = torch.cat(out).clamp_(0, 1)
    return img, (img + 0.05 * torch.randn(img.shape, device="cuda", generator=gen)).clamp_(0, 1)


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def _densify_inputs(case, seed):
    rng = np.random.default_rng(seed)
    M, n = case["prims"], case["degree"]
    # patches of mixed size and shape (scenes.mixed_shapes_scene), array-wise
    edge = 10.0 ** rng.uniform(-3, 0, M)
    high = edge * 10.0 ** rng.uniform(-3, 0, M)
    tris = np.zeros((M, 3, 3))
    tris[:, 1, 0], tris[:, 2, 0], tris[:, 2, 1] = edge, rng.uniform(-0.5, 1.5, M) * edge, high
    turn = np.linalg.qr(rng.normal(size=(M, 3, 3)))[0]
    tris = np.einsum("tck,tdk->tcd", tris, turn) + rng.uniform(-2, 2, (M, 1, 3))
    ctrl = np.einsum("ac,tcd->tad", _orders(n) / n, tris) + rng.normal(size=(M, _ncp(n), 3)) * (0.15 * edge)[:, None, None]
    sc = {"degree": n, "ctrl": ctrl, "color": rng.uniform(0, 1, ctrl.shape), "opacity": rng.uniform(0.5, 1, M),
          "r_b": rng.uniform(5e-3, 2e-2, M), "log_scale": rng.uniform(-6, -4, (M, 3)),
          "quat": rng.normal(size=(M, 4)), "bg": np.zeros(3)}
    if case["attr_res"] > 1:
        sc = scenes.with_attribute_maps(sc, case["attr_res"], seed=seed % (1 << 30))
    if case["sh"] > 0:
        sc = scenes.with_sh(sc, case["sh"], seed=seed % (1 << 30))
    grad = (rng.normal(size=ctrl.shape) * 10.0 ** rng.uniform(-5, -1, (M, 1, 1))).astype(np.float32)
    sel = np.sort(rng.permutation(M)[: max(1, M // 4)]).astype(np.int32)
    return sc, grad, sel


def prepare(case, seed):
    if case["kind"] == "loss":
        rng = np.random.default_rng(seed)
        sizes = _sizes(case, rng)
        img, target = _photos(sizes, seed)
        rd = R.Renderer(max_prims=1, max_views=1, max_pixels=1024)
        return {"case": case, "rd": rd, "img": img, "target": target,
                "cams": [{"width": w, "height": h} for w, h in sizes],
                "d": torch.empty_like(img), "loss": torch.zeros(1, device="cuda")}
    if case["kind"] == "densify":
        sc, grad, sel = _densify_inputs(case, seed)
        return {"case": case, "scene": R.scene_to_device(sc), "grad": torch.as_tensor(grad, device="cuda"),
                "sel": torch.as_tensor(sel, device="cuda")}
    rng = np.random.default_rng(seed)
    sc, centres = _scene(case, rng)
    cams = R.Cameras(_cameras(case, rng, centres))
    P = cams.pixels
    dev = R.scene_to_device(sc)
    per_px = 32 if case["scene"] == "room" else 8 if P > 1 << 18 else 24
    rd = R.Renderer(degree=case["degree"], max_prims=len(sc["ctrl"]), max_views=len(cams), max_pixels=P,
                    max_pairs=per_px * P, max_boundary_pairs=per_px * P, graph=case["graph"],
                    max_blend_pairs=24 * P if case["scene"] == "room" else 0)
    state = {"case": case, "rd": rd, "scene": dev, "cams": cams, "images": torch.empty((P, 3), device="cuda")}
    if case["kind"] in ("step", "track"):
        state["target"] = _photos([(c["width"], c["height"]) for c in cams], seed)[1]
    if case["kind"] == "step":
        params = [k for k in PARAMS if k in dev]
        if case["autograd"]:
            for k in params:
                dev[k].requires_grad_(True)
        state.update(params=params, d=torch.empty((P, 3), device="cuda"), loss=torch.zeros(1, device="cuda"),
                     grads={k: torch.empty_like(dev[k], requires_grad=False) for k in params},
                     stream=torch.cuda.Stream() if case["graph"] else None)
    if case["kind"] == "track":
        rd.forward(dev, cams, state["images"])
    torch.cuda.synchronize()
    return state


def _step(s):
    case, rd, cams, dev = s["case"], s["rd"], s["cams"], s["scene"]
    if case["autograd"]:
        img = R.render(rd, dev, cams)
        loss = R.photometric_loss(rd, img, s["target"], cams)
        grads = torch.autograd.grad(loss, [dev[k] for k in s["params"]])
        return {"images": img, "loss": loss, **{"g_" + k: g for k, g in zip(s["params"], grads)}}
    st = s["stream"]
    with torch.cuda.stream(st):
        rd.forward(dev, cams, s["images"], stream=st)
        s["loss"].zero_()
        if case["loss"] == "eq9":
            rd.l2_dssim_loss_grad(s["images"], s["target"], cams, 0.2, 1.0, s["d"], s["loss"], stream=st)
        else:
            rd.l1_loss_grad(s["images"], s["target"], 1.0 / s["images"].numel(), s["d"], s["loss"], stream=st)
        rd.backward(dev, cams, s["d"], s["grads"], stream=st)
    return {"images": s["images"], "loss": s["loss"], **{"g_" + k: g for k, g in s["grads"].items()}}


def run(state):
    kind = state["case"]["kind"]
    if kind == "step":
        return _step(state)
    if kind == "frame":
        return {"images": state["rd"].forward(state["scene"], state["cams"], state["images"])}
    if kind == "loss":
        state["loss"].zero_()
        state["rd"].l2_dssim_loss_grad(state["img"], state["target"], state["cams"], state["case"]["lam"], 1.0,
                                       state["d"], state["loss"])
        return {"loss": state["loss"], "d": state["d"]}
    if kind == "densify":
        m = R.prim_metrics(state["scene"], state["grad"])
        pieces = R.subdivide(state["scene"], state["sel"])
        return {"metrics": m, "pieces": {k: v for k, v in pieces.items() if torch.is_tensor(v)}}
    M = state["scene"]["ctrl"].shape[0]
    seen, cells = state["rd"].visibility(M)
    edges = R.edge_magnitude(state["target"], state["cams"])
    total, count = state["rd"].edge_prior(edges, M)
    return {"view_count": seen, "cell_mask": cells, "edges": edges, "edge_sum": total, "edge_count": count}


def _prims(case):
    d = case["detail"]
    return {"octa": 16, "ico": 20 * d * d, "blobs": 20 * d * d + 12 * d * max(2, 5 * d // 2),
            "room": 12 * d * d + round(2.5 * d) * (192 + 616)}[case["scene"]]


def work(case):
    """Inputs read once and outputs written once; operations of the algorithm at typical coverage (an object
    covers a quarter of a view, the room all of it; about 48 composited pairs per covered pixel, 25
    operations each forward and 73 backward; 378 per image value in the loss of Eq. 9)."""
    if case["kind"] == "loss":
        P = _pixels(case)
        return {"bytes": 36 * P, "flops": 378 * 3 * P}
    ncp = _ncp(case["degree"])
    texels, k = case["attr_res"] * (case["attr_res"] + 1) // 2, (case["sh"] + 1) ** 2 - 1
    per_prim = 4 * (6 * ncp + 2 + 7 * texels + 3 * k)
    if case["kind"] == "densify":
        M, sel = case["prims"], max(1, case["prims"] // 4)
        return {"bytes": M * (24 * ncp + 13) + sel * (4 + 5 * per_prim),
                "flops": M * 40 * ncp + sel * 4 * ncp * 30 * _ncp(case["degree"] - 1)}
    P, M = _pixels(case), _prims(case)
    if case["kind"] == "track":
        return {"bytes": 12 * P + 4 * P + 12 * P + 24 * M, "flops": 40 * P}
    covered = P * (1.0 if case["scene"] == "room" else 0.25)
    raster = case["views"] * M * TESS * TESS * 40
    if case["kind"] == "frame":
        return {"bytes": 12 * P + M * per_prim, "flops": covered * 48 * 25 + raster}
    loss = 378 * 3 * P if case["loss"] == "eq9" else 6 * P
    return {"bytes": 24 * P + 2 * M * per_prim, "flops": covered * 48 * 98 + raster + loss}


# ---------------------------------------------------------------------------
# FP64 values of the outputs, in plain torch
# ---------------------------------------------------------------------------

def _f64(x):
    return torch.as_tensor(np.asarray(x, np.float32), device="cuda").double()


def _window(x):
    """11 x 11 Gaussian window (sigma 1.5, normalised, zero outside) of [C, H, W]."""
    g = torch.exp(-torch.arange(-5, 6, device=x.device, dtype=x.dtype) ** 2 / (2 * 1.5 ** 2))
    g = (g / g.sum()).tolist()
    for dim in (1, 2):
        n = x.shape[dim]
        pad = torch.nn.functional.pad(x, (0, 0, 5, 5) if dim == 1 else (5, 5, 0, 0))
        x = sum(w * pad.narrow(dim, t, n) for t, w in enumerate(g))
    return x


def _eq9(img, target, sizes, lam):
    total, off = 0.0, 0
    for w, h in sizes:
        x, y = (t[off: off + w * h].view(h, w, 3).permute(2, 0, 1) for t in (img, target))
        off += w * h
        mx, my = _window(x), _window(y)
        vx, vy, cov = _window(x * x) - mx * mx, _window(y * y) - my * my, _window(x * y) - mx * my
        c1, c2 = 0.01 ** 2, 0.03 ** 2
        ssim = (2 * mx * my + c1) * (2 * cov + c2) / ((mx * mx + my * my + c1) * (vx + vy + c2))
        total = total + (1 - lam) * ((x - y) ** 2).mean() + lam * (1 - ssim.mean())
    return total


def _exact_loss(case, seed):
    sizes = _sizes(case, np.random.default_rng(seed))
    img, target = _photos(sizes, seed)
    grads, total, off = [], 0.0, 0
    for w, h in sizes:
        x = img[off: off + w * h].double().requires_grad_(True)
        value = _eq9(x, target[off: off + w * h].double(), [(w, h)], case["lam"])
        grads.append(torch.autograd.grad(value, x)[0])
        total, off = total + float(value.detach()), off + w * h
    return {"loss": torch.tensor([total], dtype=torch.float64), "d": torch.cat(grads)}


def _exact_densify(case, seed):
    sc, grad, sel = _densify_inputs(case, seed)
    n, M = case["degree"], case["prims"]
    ijk = _orders(n).astype(int)
    fact = np.array([math.factorial(k) for k in range(n + 1)], np.float64)
    ctrl, color = _f64(sc["ctrl"]), _f64(sc["color"])

    def at(net, bary):  # the patch at one barycentric point
        b = [math.factorial(n) / (fact[i] * fact[j] * fact[k]) * bary[0] ** i * bary[1] ** j * bary[2] ** k
             for i, j, k in ijk]
        return torch.einsum("a,mad->md", torch.tensor(b, dtype=torch.float64, device="cuda"), net)

    h = 0.5
    U, V, W = (at(ctrl, b) for b in ((1, 0, 0), (0, 1, 0), (0, 0, 1)))
    uv, uw, vw = (at(ctrl, b) for b in ((h, h, 0), (h, 0, h), (0, h, h)))
    area = sum(0.5 * torch.linalg.norm(torch.linalg.cross(b - a, c - a), dim=1)
               for a, b, c in ((U, uv, uw), (uv, V, vw), (uw, vw, W), (vw, uw, uv)))
    # bounding rectangle in the corners' plane, first axis along the longest corner edge
    corners = torch.stack([U, V, W], 1)
    edges = corners.roll(-1, 1) - corners
    first = torch.linalg.norm(edges, dim=2).argmax(1)
    rows = torch.arange(M, device="cuda")
    x = edges[rows, first] / torch.linalg.norm(edges[rows, first], dim=1, keepdim=True)
    z = torch.linalg.cross(V - U, W - U)
    y = torch.linalg.cross(z / torch.linalg.norm(z, dim=1, keepdim=True), x)
    rel = ctrl - corners[rows, first][:, None]
    ext = [torch.einsum("mad,md->ma", rel, ax) for ax in (x, y)]
    ext = torch.stack([e.amax(1) - e.amin(1) for e in ext])
    mean = torch.linalg.norm(_f64(grad), dim=2).mean(1)

    # pieces: the polar form at (A x i, B x j, C x k), one de Casteljau level per argument
    slot = {tuple(t): a for a, t in enumerate(ijk.tolist())}
    pieces = (((1, 0, 0), (h, h, 0), (h, 0, h)), ((h, h, 0), (0, 1, 0), (0, h, h)), ((h, 0, h), (0, h, h), (0, 0, 1)),
              ((0, h, h), (h, 0, h), (h, h, 0)))
    at_sel = torch.as_tensor(sel, device="cuda").long()

    def polar(net, args):
        net = {t: net[:, a] for t, a in slot.items()}
        for level, (u, v, w) in enumerate(args):
            d = n - 1 - level
            net = {(i, j, d - i - j): u * net[i + 1, j, d - i - j] + v * net[i, j + 1, d - i - j]
                   + w * net[i, j, d - i - j + 1] for i in range(d + 1) for j in range(d + 1 - i)}
        return net[0, 0, 0]

    def split(net):
        return torch.stack([torch.stack([polar(net[at_sel], [A] * i + [B] * j + [C] * k) for i, j, k in ijk], 1)
                            for A, B, C in pieces], 1).flatten(0, 1)

    res = case["attr_res"]

    def texels(maps, width):  # the parent's interpolated map at the nodes of each piece's map
        maps = _f64(maps).view(M, -1, width)[at_sel]
        if res == 1:
            return maps[:, 0].repeat_interleave(4, 0)
        m = res - 1
        where = {tuple(t): a for a, t in enumerate(_orders(m).astype(int).tolist())}
        out = []
        for piece in pieces:
            for node in _orders(m) / m:
                u, v, _ = (sum(node[c] * piece[c][k] for c in range(3)) * m for k in range(3))
                a, b = min(int(u), m - 1), min(int(v), m - 1)
                a = min(a, m - 1 - b)
                fu, fv = u - a, v - b
                if fu + fv <= 1:
                    terms = (((a, b), 1 - fu - fv), ((a + 1, b), fu), ((a, b + 1), fv))
                else:
                    terms = (((a + 1, b + 1), fu + fv - 1), ((a + 1, b), 1 - fv), ((a, b + 1), 1 - fu))
                out.append(sum(maps[:, where[i, j, m - i - j]] * w for (i, j), w in terms if w))
        return torch.stack(out, 1).view(4 * len(sel), -1, width)

    out = {"ctrl": split(ctrl), "color": split(color),
           **{k: _f64(sc[k])[at_sel].repeat_interleave(4, 0) for k in ("opacity", "r_b")},
           "log_scale": texels(sc["log_scale"], 3), "quat": texels(sc["quat"], 4)}
    if case["sh"]:
        out["sh"] = _f64(sc["sh"])[at_sel].repeat_interleave(4, 0)
    return {"metrics": {"area": area, "aspect": ext.amax(0) / ext.amin(0), "flags": None, "grad": mean},
            "pieces": out}


def _exact_edges(case, seed):
    rng = np.random.default_rng(seed)
    _, centres = _scene(case, rng)
    sizes = [(c["width"], c["height"]) for c in _cameras(case, rng, centres)]
    target, out, off = _photos(sizes, seed)[1], [], 0
    for w, h in sizes:
        c = target[off: off + w * h].double().view(h, w, 3)
        off += w * h
        y = 255 * (0.299 * c[..., 0] + 0.587 * c[..., 1] + 0.114 * c[..., 2])
        y = torch.nn.functional.pad(y[None, None], (1, 1, 1, 1), mode="replicate")[0, 0]
        sx, sy = y[:, 2:] - y[:, :-2], y[2:] - y[:-2]
        gx = sx[:-2] + 2 * sx[1:-1] + sx[2:]
        gy = sy[:, :-2] + 2 * sy[:, 1:-1] + sy[:, 2:]
        out.append((gx * gx + gy * gy).sqrt().reshape(-1))
    return {"view_count": None, "cell_mask": None, "edges": torch.cat(out), "edge_sum": None, "edge_count": None}


def _bernstein(n, uv):
    u, v = uv.unbind(-1)
    w = 1 - u - v
    return torch.stack([math.factorial(n) / (math.factorial(i) * math.factorial(j) * math.factorial(k))
                        * u ** i * v ** j * w ** k for i, j, k in _orders(n).astype(int).tolist()], -1)


def _raster(ctrl, n, cam, W, H):
    """(primitive or -1, u, v) of every pixel of one view: the nearest flat triangle of the level-TESS lattices,
    vertices on the 1/256-pixel grid, perspective-correct depth and parameters."""
    grid = [(a, b) for a in range(TESS + 1) for b in range(TESS + 1 - a)]
    slot = {ab: k for k, ab in enumerate(grid)}
    tri = [(slot[a, b], slot[a + 1, b], slot[a, b + 1]) for a in range(TESS) for b in range(TESS - a)]
    tri += [(slot[a + 1, b], slot[a + 1, b + 1], slot[a, b + 1]) for a in range(TESS) for b in range(TESS - 1 - a)]
    uv = torch.tensor(grid, dtype=torch.float64, device="cuda") / TESS
    cp = torch.einsum("va,mad->mvd", _bernstein(n, uv), ctrl) @ cam["R"].T + cam["t"]
    xy = torch.round((cam["f"] * cp[..., :2] / cp[..., 2:] + cam["c"]) * 256)
    tri = torch.tensor(tri, device="cuda")
    p, z = xy[:, tri].flatten(0, 1), cp[..., 2][:, tri].flatten(0, 1)
    prim = torch.arange(len(ctrl), device="cuda").repeat_interleave(len(tri))
    tuv = uv[tri].repeat(len(ctrl), 1, 1)
    area = (p[:, 1, 0] - p[:, 0, 0]) * (p[:, 2, 1] - p[:, 0, 1]) - (p[:, 1, 1] - p[:, 0, 1]) * (p[:, 2, 0] - p[:, 0, 0])
    flip = (area < 0)[:, None]
    order = torch.where(flip, torch.tensor([0, 2, 1], device="cuda"), torch.tensor([0, 1, 2], device="cuda"))
    p, z = p.gather(1, order[..., None].expand(-1, -1, 2)), z.gather(1, order)
    tuv = tuv.gather(1, order[..., None].expand(-1, -1, 2))
    lo = torch.ceil(p.amin(1) / 256).clamp(min=0)
    hi = torch.minimum(torch.floor(p.amax(1) / 256), torch.tensor([W - 1.0, H - 1.0], device="cuda", dtype=torch.float64))
    wide, high = ((hi - lo + 1).clamp(min=0).long() * (area != 0)[:, None]).unbind(1)
    count = wide * high
    frag = torch.arange(len(p), device="cuda").repeat_interleave(count)
    k = torch.arange(len(frag), device="cuda") - (count.cumsum(0) - count)[frag]
    px, py = lo[frag, 0].long() + k % wide[frag], lo[frag, 1].long() + k // wide[frag]
    q, pf = torch.stack([px, py], 1).double() * 256, p[frag]
    e, inside = [], torch.ones(len(frag), dtype=torch.bool, device="cuda")
    for a, b in ((1, 2), (2, 0), (0, 1)):
        d = pf[:, b] - pf[:, a]
        v = d[:, 0] * (q[:, 1] - pf[:, a, 1]) - d[:, 1] * (q[:, 0] - pf[:, a, 0])
        own = (d[:, 1] < 0) | ((d[:, 1] == 0) & (d[:, 0] > 0))
        inside &= (v > 0) | ((v == 0) & own)
        e.append(v)
    e = (torch.stack(e, 1) / z[frag])[inside]
    frag, pix = frag[inside], (py * W + px)[inside]
    near = torch.sort(e.sum(1) / area[frag].abs(), descending=True, stable=True).indices
    near = near[torch.sort(pix[near], stable=True).indices]
    pix_s = pix[near]
    first = near[torch.cat([torch.ones(1, dtype=torch.bool, device="cuda"), pix_s[1:] != pix_s[:-1]])]
    ids = torch.full((W * H,), -1, dtype=torch.long, device="cuda")
    out = torch.zeros((W * H, 2), dtype=torch.float64, device="cuda")
    ids[pix[first]] = prim[frag[first]]
    out[pix[first]] = (tuv[frag[first]] * e[first][..., None]).sum(1) / e[first].sum(1, keepdim=True)
    return ids, out


def _blend(par, n, cam, W, H):
    """The image of one view, differentiable in the parameters with ids, (u, v) and the boundary set held."""
    with torch.no_grad():
        ids, uv = _raster(par["ctrl"], n, cam, W, H)
        im = ids.view(H, W)
        differ = torch.zeros((H, W), dtype=torch.bool, device="cuda")
        differ[:, 1:] |= im[:, 1:] != im[:, :-1]
        differ[:, :-1] |= im[:, 1:] != im[:, :-1]
        differ[1:] |= im[1:] != im[:-1]
        differ[:-1] |= im[1:] != im[:-1]
        fg = (ids >= 0).nonzero()[:, 0]
        edge = differ.reshape(-1)[fg]
    g = ids[fg]
    B = _bernstein(n, uv[fg])
    t = torch.einsum("fa,fad->fd", B, par["ctrl"][g]) @ cam["R"].T + cam["t"]
    col = torch.einsum("fa,fad->fd", B, par["color"][g])
    mu = cam["f"] * t[:, :2] / t[:, 2:] + cam["c"]
    q = par["quat"][g]
    r, x, y, z = (q / torch.linalg.norm(q, dim=1, keepdim=True)).unbind(1)
    rot = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - r * z), 2 * (x * z + r * y),
                       2 * (x * y + r * z), 1 - 2 * (x * x + z * z), 2 * (y * z - r * x),
                       2 * (x * z - r * y), 2 * (y * z + r * x), 1 - 2 * (x * x + y * y)], 1).view(-1, 3, 3)
    m3 = rot * par["log_scale"][g].exp()[:, None]
    zero = torch.zeros_like(t[:, 0])
    jac = torch.stack([cam["f"] / t[:, 2], zero, -cam["f"] * t[:, 0] / t[:, 2] ** 2,
                       zero, cam["f"] / t[:, 2], -cam["f"] * t[:, 1] / t[:, 2] ** 2], 1).view(-1, 2, 3)
    half = jac @ cam["R"] @ m3
    cov = half @ half.transpose(1, 2) + 0.3 * torch.eye(2, dtype=torch.float64, device="cuda")
    con = torch.linalg.inv(cov)
    op = par["opacity"][g]
    bpt, bsig, bprim = mu[edge], 3 * cam["f"] * par["r_b"][g][edge] / t[edge, 2], g[edge]
    with torch.no_grad():
        reach = (2 * torch.log((op * 255).clamp(min=1))[:, None] * torch.stack([cov[:, 0, 0], cov[:, 1, 1]], 1)).sqrt()
    rows = []
    size = 16
    for y0 in range(0, H, size):
        for x0 in range(0, W, size):
            x1, y1 = min(x0 + size, W), min(y0 + size, H)
            lo = torch.tensor([x0, y0], dtype=torch.float64, device="cuda")
            hi = torch.tensor([x1 - 1, y1 - 1], dtype=torch.float64, device="cuda")
            with torch.no_grad():
                hit = ((mu + reach >= lo) & (mu - reach <= hi)).all(1).nonzero()[:, 0]
                hit = hit[torch.sort(t[hit, 2], stable=True).indices]
                near = ((bpt + bsig[:, None] > lo) & (bpt - bsig[:, None] < hi)).all(1).nonzero()[:, 0]
                px = torch.stack(torch.meshgrid(torch.arange(y0, y1, device="cuda"), torch.arange(x0, x1, device="cuda"),
                                                indexing="ij")[::-1], -1).view(-1, 2)
                pid = ids[px[:, 1] * W + px[:, 0]]
                px = px.double()
                names, slot = torch.unique(g[hit], return_inverse=True)
                if len(hit):
                    at = torch.searchsorted(names, bprim[near]).clamp(max=len(names) - 1)
                    keep = names[at] == bprim[near]
                    near, at = near[keep], at[keep]
            if not len(hit):  # background
                continue
            d, K = px[:, None] - mu[hit], con[hit]
            G = torch.exp(-0.5 * (K[:, 0, 0] * d[..., 0] ** 2 + 2 * K[:, 0, 1] * d[..., 0] * d[..., 1]
                                  + K[:, 1, 1] * d[..., 1] ** 2))
            # Eq. 6-7: the most influential boundary point of each primitive, per pixel
            rho = torch.linalg.norm(px[:, None] - bpt[near], dim=2) / bsig[near]
            low = torch.ones((len(px), len(names)), dtype=torch.float64, device="cuda")
            if len(near):
                low = low.scatter_reduce(1, at.expand(len(px), -1), rho, "amin", include_self=True)
            gamma = 2 ** (low - 1)
            w = torch.where(pid[:, None] == names, gamma, 1 - gamma)[:, slot]
            alpha = (op[hit] * w * G).clamp(max=0.99)
            alpha = torch.where(alpha >= 1 / 255, alpha, torch.zeros_like(alpha))
            after = torch.cumprod(1 - alpha, 1)
            alpha = torch.where(after >= 1e-4, alpha, torch.zeros_like(alpha))
            T = torch.cumprod(torch.cat([torch.ones_like(alpha[:, :1]), 1 - alpha], 1), 1)[:, :-1]
            rows.append(((px[:, 1] * W + px[:, 0]).long(), (T * alpha) @ col[hit]))
    where = torch.cat([r for r, _ in rows])
    return torch.zeros((W * H, 3), dtype=torch.float64, device="cuda").index_put((where,), torch.cat([c for _, c in rows]))


def _exact_render(case, seed):
    rng = np.random.default_rng(seed)
    sc, centres = _scene(case, rng)
    cams = _cameras(case, rng, centres)
    par = {k: _f64(sc[k]).requires_grad_(True) for k in PARAMS if k in sc}
    images = []
    for c in cams:
        cam = {"R": _f64(c["R"]), "t": _f64(c["t"]), "f": float(c["fx"]), "c": _f64([c["cx"], c["cy"]])}
        images.append(_blend(par, case["degree"], cam, c["width"], c["height"]))
    img = torch.cat(images)
    if case["kind"] == "frame":
        return {"images": img.detach()}
    sizes = [(c["width"], c["height"]) for c in cams]
    target = _photos(sizes, seed)[1].double()
    loss = _eq9(img, target, sizes, 0.2)
    grads = torch.autograd.grad(loss, list(par.values()))
    return {"images": img.detach(), "loss": loss.detach(), **{"g_" + k: v for k, v in zip(par, grads)}}


def exact(case, seed):
    """The outputs of run() in FP64, or None where plain torch takes too long (renders of more than about
    60,000 pixels), and for attribute maps and SH colour."""
    if case["kind"] == "loss":
        return _exact_loss(case, seed)
    if case["kind"] == "densify":
        return _exact_densify(case, seed)
    if case["kind"] == "track":
        return _exact_edges(case, seed)
    small = _pixels(case) <= 60_000 and _prims(case) <= 4000
    if not small or case["attr_res"] > 1 or case["sh"] or (case["kind"] == "step" and case["loss"] != "eq9"):
        return None
    return _exact_render(case, seed)
