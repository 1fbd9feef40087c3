"""Timed cases of the library's main path: the calls a pose-inference program makes, each through
the public Python entry points, over the sizes and options of the repository's workloads.

A case is a dict of plain values; ``prepare`` builds the scene, the observation and the inputs it
names, ``run`` makes one call (or the two or three calls that belong together), ``exact`` restates
the result in 64-bit torch from the geometry alone: every object of these scenes is a union of
lattice cells (or a flat table), so the depth along a pixel's ray is the nearest lattice plane
crossing that bounds an occupied cell. The observations are rendered the same way, so no input
comes from the code that is timed.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2312_08715_gb300 import b3d, synth

DEV = "cuda"
F64 = torch.float64


# ------------------------------------------------------------------------------------------
# the cases
# ------------------------------------------------------------------------------------------

def listed():
    return [
        # the single-object configuration: 10^3 grid cells, the call whose launch and host cost count
        dict(name="score_single_64x48", kind="score", scene="single", width=64, height=48, n_obj=1, vox=500, n=1000,
             lik=0, half_window=1, miss_mode=0, spread=0.05, tuned=0),
        # one coarse-to-fine stage of the tabletop parse (9^3 translations x 200 rotations), with the
        # launch shape a program keeps after autotuning it once
        dict(name="score_tabletop_160x120", kind="score", scene="tabletop", width=160, height=120, n_obj=5, vox=4500,
             n=145800, lik=0, half_window=1, miss_mode=0, spread=0.08, tuned=1),
        # a finer stage at the image size of the tracking sessions, library defaults
        dict(name="score_320x240", kind="score", scene="tabletop", width=320, height=240, n_obj=3, vox=4500, n=31250,
             lik=0, half_window=1, miss_mode=0, spread=0.025, tuned=0),
        # the smooth likelihood over a 5x5 window on an image of odd size
        dict(name="score_smooth_150x113", kind="score", scene="tabletop", width=150, height=113, n_obj=4, vox=3000,
             n=16001, lik=1, half_window=2, miss_mode=0, spread=0.025, tuned=0),
        # eight scenes of uneven size in one launch (the batched form)
        dict(name="score_multi_8", kind="multi", scene="tabletop", scenes=8, width=320, height=240, n_obj=3, vox=4000,
             n=6000, lik=0, half_window=1, miss_mode=0, spread=0.04),
        # one tracking step: a new depth frame, then the enumeration around the last estimate
        dict(name="track_320x240", kind="track", scene="tabletop", width=320, height=240, n_obj=3, vox=4500, n=6250,
             stages=1, particles=16, lik=0, half_window=1, miss_mode=0),
        # depth and triangle-id images of particles
        dict(name="render_ids_160x120", kind="render", scene="tabletop", width=160, height=120, n_obj=5, vox=4500,
             n=2048, spread=0.025),
        # the render-then-score form, images in device memory
        dict(name="render_score_160x120", kind="materialised", scene="tabletop", width=160, height=120, n_obj=5,
             vox=4500, n=20000, lik=0, half_window=1, miss_mode=0, spread=0.05),
        # one stage of camera-pose tracking at the largest size of its table
        dict(name="camera_200x200", kind="camera", scene="camera", width=200, height=200, n_obj=4, vox=12000, n=2048,
             lik=0, half_window=1, miss_mode=0),
        # forward and backward of the smooth likelihood for a set of particles (one refinement step)
        dict(name="grad_256_160x120", kind="grad", scene="tabletop", width=160, height=120, n_obj=5, vox=4500, n=256,
             lik=1, half_window=2, miss_mode=0, spread=0.005),
        # hierarchical noise: 4 x 4 settings per hypothesis
        dict(name="noise_160x120", kind="noise", scene="tabletop", width=160, height=120, n_obj=5, vox=4500, n=8192,
             lik=0, half_window=1, miss_mode=0, spread=0.05, n_radius=4, n_pout=4),
        # normalise and resample the scores of one stage
        dict(name="resample_145800", kind="resample", n=145800, particles=100),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["score", "score", "score", "multi", "track", "render", "materialised", "camera", "grad", "noise",
                       "resample"])
    if kind == "resample":
        return dict(kind=kind, n=int(_log(rng, 1000, 400000)), particles=int(_log(rng, 1, 1000)))
    if kind == "camera":
        size = int(_log(rng, 25, 201))
        n = int(_log(rng, 256, 4096)) if size < 140 else int(_log(rng, 256, 2048))
        return dict(kind=kind, scene="camera", width=size, height=size, n_obj=4, vox=int(_log(rng, 4000, 13000)), n=n,
                    lik=0, half_window=1, miss_mode=0)
    w = int(_log(rng, 64, 330))
    h = max(48, int(w * 0.75) + rng.randrange(-3, 4))
    vox = int(_log(rng, 600, 16000))
    c = dict(kind=kind, scene="tabletop", width=w, height=h, n_obj=rng.randrange(1, 7), vox=vox)
    # hypotheses: up to a budget of footprint pixels well below that of the largest listed case
    foot = max(_footprint(c), 150.0)
    most = {"score": 6e7, "multi": 1.5e7, "track": 2.5e7, "render": 1.5e6, "materialised": 1e7, "grad": 1e6,
            "noise": 5e6}[kind] / foot
    if kind in ("render", "materialised"):
        most = min(most, {"render": 4e7, "materialised": 3.5e8}[kind] / (w * h))
    lo = {"score": 500, "multi": 300, "track": 1000, "render": 16, "materialised": 256, "grad": 16, "noise": 256}[kind]
    c["n"] = int(_log(rng, lo, max(2 * lo, min(most, 145800))))
    if kind in ("score", "multi", "noise"):
        c["lik"] = 1 if rng.random() < 0.3 else 0
    elif kind != "render":
        c["lik"] = 1 if kind == "grad" else 0
    if kind != "render":
        c["half_window"] = rng.choice([1, 1, 1, 2, 2]) if kind != "score" else rng.choice([1, 1, 1, 1, 2, 2, 3])
        c["miss_mode"] = 1 if kind in ("score", "multi") and rng.random() < 0.2 else 0
    if kind != "track":
        c["spread"] = round(_log(rng, 0.004, 0.08), 4)
    if kind == "score":
        c["tuned"] = rng.randrange(2)
    if kind == "multi":
        c["scenes"] = rng.randrange(2, 9)
        c["n"] = max(200, c["n"] // 3)
    if kind == "track":
        c["stages"], c["particles"] = rng.randrange(1, 4), int(_log(rng, 1, 128))
    if kind == "noise":
        c["n_radius"], c["n_pout"] = rng.randrange(1, 5), rng.randrange(1, 5)
    return c


# ------------------------------------------------------------------------------------------
# scenes
# ------------------------------------------------------------------------------------------

def _scene(case, seed):
    """(synth.Scene, slot, grid frame or None): camera_scene poses are world poses."""
    W, H = case["width"], case["height"]
    trial = int(seed) % (1 << 28)
    v = case["vox"]
    if case["scene"] == "single":
        wl = synth.single_object_workload(trial)
        return wl.scene, 0, np.eye(3, dtype=np.float32), None
    if case["scene"] == "camera":
        video = synth.camera_video(trial, W, n_frames=1, vox_lo=int(0.7 * v), vox_hi=int(1.4 * v))
        return video.scene, -1, None, video.cam_from_world[0]
    wl = synth.tabletop_workload(trial, n_objects=case["n_obj"], width=W, height=H, f=0.9375 * W, vox_lo=int(0.6 * v),
                                 vox_hi=int(1.5 * v), seed_base=11000)
    return wl.scene, wl.slot, wl.grid_frame, None


def _lattice(mesh):
    """Plane coordinates per axis and the occupied cells of a union of boxes of one lattice
    (8 vertices a box); a flat mesh keeps two extents and has no cells."""
    v = mesh.verts.astype(np.float64)
    axes = [np.unique(v[:, k]) for k in range(3)]
    if len(axes[2]) == 1:
        return axes, None
    lo = v.reshape(-1, 8, 3).min(1)
    idx = np.stack([np.searchsorted(axes[k], lo[:, k]) for k in range(3)], 1)
    occ = np.zeros([len(a) + 1 for a in axes], dtype=bool)  # one empty cell of margin on each side
    occ[idx[:, 0] + 1, idx[:, 1] + 1, idx[:, 2] + 1] = True
    return axes, torch.as_tensor(occ, device=DEV)


def _rays(cam, x, y):
    fx, fy = float(np.float32(cam.fx)), float(np.float32(cam.fy))
    cx, cy = float(np.float32(cam.cx)), float(np.float32(cam.cy))
    return (x.to(F64) + 0.5 - cx) / fx, (y.to(F64) + 0.5 - cy) / fy


def _inv3(A):
    """Inverses of 3x3 matrices [n, 3, 3] by their adjugates."""
    r = A.unbind(1)
    adj = torch.stack([torch.linalg.cross(r[1], r[2]), torch.linalg.cross(r[2], r[0]), torch.linalg.cross(r[0], r[1])], 2)
    return adj / (r[0] * adj[:, :, 0]).sum(1)[:, None, None]


def _cast(mesh, poses, rx, ry, far, want_axis=False):
    """Depth of `mesh` at poses [B, 4, 4] along rays (rx, ry, 1) [B, P], `far` where it is missed
    (64-bit); with want_axis also the lattice axis of the face that is hit (-1: none)."""
    axes, occ = mesh
    M = _inv3(poses.to(F64)[:, :3, :3])
    o = -(M @ poses.to(F64)[:, :3, 3:])  # [B, 3, 1]
    d = [M[:, k, 0:1] * rx + M[:, k, 1:2] * ry + M[:, k, 2:3] for k in range(3)]
    best = torch.full_like(rx, far)
    hit_axis = torch.full(rx.shape, -1, dtype=torch.int8, device=rx.device) if want_axis else None
    coords = [torch.as_tensor(a, device=rx.device) for a in axes]
    for a in range(3):
        if occ is None and a != 2:
            continue
        b, c = (a + 1) % 3, (a + 2) % 3
        inv = 1.0 / d[a]
        for p in range(len(axes[a])):
            t = (coords[a][p] - o[:, a]) * inv
            q = [o[:, k] + t * d[k] for k in (b, c)]
            inside = (t > 0) & (t < best)
            for k, u in zip((b, c), q):
                inside &= (u >= coords[k][0]) & (u <= coords[k][-1])
            if occ is not None:
                jb, jc = (torch.searchsorted(coords[k], u.contiguous(), right=True) for k, u in zip((b, c), q))
                layer = (occ.select(a, p) | occ.select(a, p + 1))  # [b', c'] in ascending axis order
                if b > c:
                    layer = layer.t()
                jb, jc = (j.clamp(1, len(axes[k]) - 1) for j, k in zip((jb, jc), (b, c)))
                inside &= layer[jb, jc]
            best = torch.where(inside, t, best)
            if want_axis:
                hit_axis = torch.where(inside, torch.full_like(hit_axis, a), hit_axis)
    return (best, hit_axis) if want_axis else best


def _image_rays(cam):
    y, x = torch.meshgrid(torch.arange(cam.height, device=DEV), torch.arange(cam.width, device=DEV), indexing="ij")
    return _rays(cam, x.reshape(1, -1), y.reshape(1, -1))


def _fixed_depth(scene, lattices, poses, skip):
    """Depth image [H, W] of every object but `skip` (64-bit)."""
    cam = scene.camera
    far = float(np.float32(cam.far))
    rx, ry = _image_rays(cam)
    best = torch.full_like(rx, far)
    for k, m in enumerate(lattices):
        if k != skip:
            P = torch.as_tensor(np.asarray(poses[k], np.float64), device=DEV)[None]
            best = torch.minimum(best, _cast(m, P, rx, ry, far))
    return best.reshape(cam.height, cam.width)


def _observe(scene, lattices, poses, seed):
    """Observed depth [H, W] float32: 2 mm noise on surfaces, 10% uniform outliers."""
    clean = _fixed_depth(scene, lattices, poses, -1).cpu().numpy()
    rng = np.random.default_rng([77, int(seed)])
    draws = synth.noise_draws(rng, scene.camera.height, scene.camera.width)
    return torch.as_tensor(synth.corrupt_depth(clean, scene.camera.far, draws), device=DEV)


def _exp_rot(r):
    """Rotation matrices [n, 3, 3] of rotation vectors [n, 3] (64-bit; Rodrigues' formula)."""
    K = torch.zeros((r.shape[0], 3, 3), dtype=F64, device=r.device)
    K[:, 0, 1], K[:, 0, 2], K[:, 1, 2] = -r[:, 2], r[:, 1], -r[:, 0]
    K = K - K.transpose(1, 2)
    a = r.norm(dim=1).clamp(min=1e-12)[:, None, None]
    eye = torch.eye(3, dtype=F64, device=r.device)
    return eye + torch.sin(a) / a * K + (1 - torch.cos(a)) / (a * a) * (K @ K)


def _poses(n, centre, frame, spread, max_deg, seed):
    """n poses [n, 4, 4] float32 around `centre`: 9^3 translation cells over +- spread in the grid
    frame for each of a set of rotations, rotation by rotation as a coarse-to-fine stage lists them."""
    g = torch.Generator().manual_seed(int(seed) + 5)
    n_rot = -(-n // 729)
    r = torch.randn((n_rot, 3), generator=g, dtype=F64)
    r = r / r.norm(dim=1, keepdim=True) * math.radians(max_deg) * torch.rand((n_rot, 1), generator=g, dtype=F64) ** (1 / 3)
    R = _exp_rot(r.to(DEV))
    i = torch.arange(n, device=DEV)
    cell = i % 729
    off = torch.stack([cell // 81, (cell // 9) % 9, cell % 9], 1).to(F64) - 4.0
    C = torch.as_tensor(np.asarray(centre, np.float64), device=DEV)
    G = torch.as_tensor(np.asarray(frame, np.float64), device=DEV)
    P = torch.zeros((n, 4, 4), dtype=F64, device=DEV)
    P[:, :3, :3] = (C[:3, :3] @ R)[i // 729]
    P[:, :3, 3] = C[:3, 3] + (off * (spread / 4.0)) @ G.T
    P[:, 3, 3] = 1.0
    return P.float()


def _camera_poses(n, base, seed):
    """n camera_from_world poses: rotations about the world origin of up to 1 degree."""
    g = torch.Generator().manual_seed(int(seed) + 6)
    r = torch.randn((n, 3), generator=g, dtype=F64)
    r = r / r.norm(dim=1, keepdim=True) * math.radians(1.0) * torch.rand((n, 1), generator=g, dtype=F64) ** (1 / 3)
    B = torch.as_tensor(np.asarray(base, np.float64), device=DEV)
    P = B.repeat(n, 1, 1)
    P[:, :3, :3] = B[:3, :3] @ _exp_rot(r.to(DEV))
    return P.float()


def _lik(case):
    smooth = case["lik"] == 1
    return dict(kind=case["lik"], radius=0.003 if smooth else 0.005, p_outlier=0.01, half_window=case["half_window"],
                miss_mode=case["miss_mode"])


def _noise(case):
    radii = [0.002, 0.004, 0.007, 0.012][:case["n_radius"]]
    pouts = [0.005, 0.02, 0.1, 0.3][:case["n_pout"]]
    return radii, pouts


def _inputs(case, seed):
    """Everything a call needs but the library's own objects, from the seed alone."""
    scene, slot, frame, cam0 = _scene(case, seed)
    lattices = [_lattice(m) for m in scene.meshes]
    rng = np.random.default_rng([3, int(seed)])
    if case["scene"] == "camera":
        true = np.stack([cam0.astype(np.float64) @ P for P in scene.poses.astype(np.float64)])
        small = _exp_rot(torch.as_tensor(rng.normal(size=(1, 3)) * 0.004, device=DEV))[0].cpu().numpy()
        base = np.asarray(cam0, np.float64).copy()
        base[:3, :3] = base[:3, :3] @ small  # the search starts near the true camera
        poses = _camera_poses(case["n"], base, seed)
        return dict(scene=scene, lattices=lattices, slot=-1, obs=_observe(scene, lattices, true, seed), poses=poses)
    obs = _observe(scene, lattices, scene.poses, seed)
    centre = scene.poses[slot].astype(np.float64).copy()
    near = case.get("spread", 0.02) * 0.25
    centre[:3, 3] += np.asarray(frame, np.float64) @ rng.uniform(-near, near, size=3)
    centre[:3, :3] = centre[:3, :3] @ synth.yaw(math.radians(rng.uniform(-3, 3)))
    out = dict(scene=scene, lattices=lattices, slot=slot, obs=obs, centre=centre.astype(np.float32), frame=frame)
    if case["kind"] != "track":
        out["poses"] = _poses(case["n"], centre, frame, case["spread"], 10.0 if case["spread"] > 0.01 else 2.0, seed)
    return out


def _context(inp):
    ctx = b3d.Context(0)
    sc = inp["scene"]
    ids = [ctx.load_mesh(m, closed=m.faces.shape[0] % 12 == 0) for m in sc.meshes]
    ctx.set_scene(sc.camera, ids, sc.poses, inp["obs"])
    return ctx


def _multi_cases(case):
    """The scenes of a batched call: widths, object counts, sizes and hypotheses fall off unevenly."""
    out = []
    for k in range(case["scenes"]):
        s = 0.5 ** (2.0 * k / max(case["scenes"] - 1, 1))
        w = max(64, int(case["width"] * s) - k)
        out.append(dict(case, width=w, height=max(48, int(case["height"] * s) - 2 * k), n_obj=1 + (case["n_obj"] + k) % 4,
                        vox=max(500, int(case["vox"] * (1 + k % 3) / 2)), n=max(100, case["n"] // (1 + (3 * k) % 5))))
    return out


# ------------------------------------------------------------------------------------------
# prepare and run
# ------------------------------------------------------------------------------------------

def prepare(case, seed):
    kind = case["kind"]
    if kind == "resample":
        ll = synth.random_ll(np.random.default_rng([9, int(seed)]), case["n"])
        return dict(kind=kind, ctx=b3d.Context(0), ll=torch.as_tensor(ll, device=DEV), m=case["particles"],
                    seed=int(seed) + 1)
    if kind == "multi":
        owner, items, ctxs = b3d.Context(0), [], []
        outs = []
        for k, c in enumerate(_multi_cases(case)):
            inp = _inputs(c, seed + 1000003 * k)
            ctx = _context(inp)
            ctxs.append((ctx, inp["poses"]))
            outs.append(torch.zeros(c["n"], dtype=torch.float32, device=DEV))
            items.append((ctx.h, inp["slot"], c["n"], inp["poses"], outs[-1]))
        return dict(kind=kind, ctx=owner, items=items, outs=outs, keep=ctxs, lik=b3d.lik_params(**_lik(case)))
    inp = _inputs(case, seed)
    ctx = _context(inp)
    st = dict(kind=kind, ctx=ctx, slot=inp["slot"], obs=inp["obs"], poses=inp.get("poses"))
    if "lik" in case:
        st["lik"] = _lik(case)
    if kind == "score" and case["tuned"]:
        wide = case["width"] >= 240  # the shapes the autotuner settles on at the two image sizes
        b3d.b3d_set_tuning(ctx.h, 96, 256 if wide else 128, 0, 0, 4)
    if kind == "track":
        n_rot = max(1, case["n"] // 125)
        steps = [0.01, 0.0025, 0.0006][:case["stages"]]
        st |= dict(stages=[synth.StageSpec(5, s, 1, n_rot, math.radians(5.0 * s / 0.01)) for s in steps],
                   m=case["particles"], seed=int(seed) + 2, centre=inp["centre"], frame=inp["frame"])
    if kind == "noise":
        radii, pouts = _noise(case)
        st["grid"] = b3d.noise_grid(case["lik"], radii, pouts, case["half_window"],
                                    np.full(len(radii) * len(pouts), -math.log(len(radii) * len(pouts))))
    return st


def run(st):
    kind, ctx = st["kind"], st["ctx"]
    if kind == "score":
        return ctx.score(st["slot"], st["poses"], st["lik"])
    if kind == "multi":
        b3d.b3d_score_multi(ctx.h, st["items"], st["lik"], ctx.stream)
        return st["outs"]
    if kind == "track":
        ctx.set_observation(st["obs"])
        return ctx.enumerate_c2f(st["slot"], st["centre"], st["stages"], st["lik"], st["m"], st["seed"], st["frame"])
    if kind == "render":
        return ctx.render(st["slot"], st["poses"])
    if kind == "materialised":
        depth, _ = ctx.render(st["slot"], st["poses"], want_tid=False)
        return depth, ctx.score_depth(depth, st["lik"], slot=st["slot"])
    if kind == "camera":
        depth, _ = ctx.render_camera(st["poses"], want_tid=False)
        return depth, ctx.score_depth(depth, st["lik"])
    if kind == "grad":
        return ctx.score_grad(st["slot"], st["poses"], st["lik"])
    if kind == "noise":
        return ctx.score_noise(st["slot"], st["poses"], st["grid"])
    return ctx.lse_resample(st["ll"], st["m"], st["seed"], 0)


# ------------------------------------------------------------------------------------------
# work
# ------------------------------------------------------------------------------------------

def _footprint(case):
    """Screen pixels of an object of `vox` cells (5 mm; 1 cm for the single object) at its usual
    distance: the silhouette of a ball of that volume."""
    pitch, dist = (0.01, 0.5) if case["scene"] == "single" else (0.005, 0.6 if case["scene"] == "camera" else 0.8)
    f = case["width"] * (1.0 if case["scene"] == "camera" else 0.9375)
    return math.pi * (3.0 * case["vox"] / (4.0 * math.pi)) ** (2.0 / 3.0) * (pitch * f / dist) ** 2


def work(case):
    kind, n = case["kind"], case["n"]
    if kind == "resample":
        return dict(bytes=4.0 * n + 8.0 * case["particles"] + 4, flops=4.0 * n)
    if kind == "multi":
        parts = [work(dict(c, kind="score")) for c in _multi_cases(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    npx = case["width"] * case["height"]
    foot = min(_footprint(case), npx)
    scored = npx if kind == "camera" else foot
    window = (2 * case.get("half_window", 0) + 1) ** 2
    settings = case.get("n_radius", 1) * case.get("n_pout", 1)
    # per rendered pixel a plane's depth; per scored pixel the window's distances (8 operations each)
    # and one term per setting; the gradient visits the window twice
    flops = n * (foot * 6.0 + (0 if kind == "render" else scored * (window * 8.0 * (3.0 if kind == "grad" else 1.0) + 4.0 * settings)))
    data = 64.0 * n + 12.0 * npx
    if kind == "render":
        data += 8.0 * n * npx
    elif kind in ("materialised", "camera"):
        data += 8.0 * n * npx + 4.0 * n  # written, then read by the scorer
    elif kind == "grad":
        data += 36.0 * n
    elif kind == "noise":
        data += 4.0 * n * (settings + 1)
    elif kind == "track":
        n_st = max(1, n // 125) * 125 * case["stages"]
        flops *= n_st / n
        data = 16.0 * npx + 4.0 * n_st + 72.0 * case["particles"]
    else:
        data += 4.0 * n
    return dict(bytes=data, flops=flops)


# ------------------------------------------------------------------------------------------
# the same results in 64 bits
# ------------------------------------------------------------------------------------------

def _constants(lik, cam):
    w = lik["half_window"]
    r, p = (float(np.float32(lik[k])) for k in ("radius", "p_outlier"))
    V = cam.width * cam.height / (cam.fx * cam.fy) * (float(np.float32(cam.far)) ** 3 - float(np.float32(cam.near)) ** 3) / 3.0
    K = (2 * w + 1) ** 2
    return r, p, V, K


def _terms(depth, obs, x, y, cam, lik, settings=None):
    """l_i [B, h, w] of observed depths obs [B, h, w] at pixels x, y, given rendered depths with
    a margin of the half window on every side ([B, h + 2w, w + 2w], NaN: no point)."""
    w = lik["half_window"]
    h_, w_ = obs.shape[-2:]
    rx, ry = _rays(cam, x, y)
    ok = (obs > 0) & torch.isfinite(obs)
    qx, qy = obs * rx, obs * ry
    settings = settings or [(lik["radius"], lik["p_outlier"])]
    radii = sorted({r for r, _ in settings})
    sums = {r: torch.zeros_like(obs) for r in radii}
    for dy in range(2 * w + 1):
        for dx in range(2 * w + 1):
            z = depth[..., dy:dy + h_, dx:dx + w_]
            jx, jy = _rays(cam, x + (dx - w), y + (dy - w))
            d2 = (qx - z * jx) ** 2 + (qy - z * jy) ** 2 + (obs - z) ** 2
            for r in radii:
                r64 = float(np.float32(r))
                k = (d2 <= r64 * r64).to(F64) if lik["kind"] == 0 else torch.exp(-d2 / (2 * r64 * r64))
                sums[r] += torch.where(torch.isnan(d2), torch.zeros_like(k), k)
    out = []
    for r, p in settings:
        r64, p64, V, K = _constants(dict(lik, radius=r, p_outlier=p), cam)
        norm = 1.0 / (4.0 / 3.0 * math.pi * r64 ** 3) if lik["kind"] == 0 else (2 * math.pi * r64 * r64) ** -1.5
        out.append(torch.where(ok, torch.log(p64 / V + (1 - p64) / K * norm * sums[r]), torch.zeros_like(obs)))
    return out


def _pad(img, w):
    return torch.nn.functional.pad(img, (w, w, w, w), value=float("nan"))


def _crop_boxes(mesh, poses, cam, margin):
    """Screen boxes (x0, y0) [B] and one common size that holds the object and the margin."""
    axes, _ = mesh
    c = torch.tensor([[axes[0][i], axes[1][j], axes[2][k]] for i in (0, -1) for j in (0, -1) for k in (0, -1)], device=DEV)
    P = poses.to(F64)
    q = torch.einsum("bij,kj->bki", P[:, :3, :3], c) + P[:, None, :3, 3]
    u, v = cam.fx * q[..., 0] / q[..., 2] + cam.cx, cam.fy * q[..., 1] / q[..., 2] + cam.cy
    x0, x1 = (torch.floor(u.amin(1)) - margin).long(), (torch.ceil(u.amax(1)) + margin).long()
    y0, y1 = (torch.floor(v.amin(1)) - margin).long(), (torch.ceil(v.amax(1)) + margin).long()
    w = min(int((x1 - x0).amax()) + 1, cam.width)
    h = min(int((y1 - y0).amax()) + 1, cam.height)
    return x0.clamp(0, cam.width - w), y0.clamp(0, cam.height - h), w, h


def _exact_scores(case, seed, settings=None, limit=1.6e9):
    """Sum of l_i of every hypothesis (per setting), by the crop around the object's screen box:
    the pixels outside it keep the fixed objects' terms."""
    inp = _inputs(case, seed)
    sc, slot, cam, poses = inp["scene"], inp["slot"], inp["scene"].camera, inp["poses"]
    lik, far = _lik(case), float(np.float32(cam.far))
    w = lik["half_window"]
    bg = _fixed_depth(sc, inp["lattices"], sc.poses, slot)
    gap = float("nan") if lik["miss_mode"] == 1 else far
    bgz = torch.where(bg >= far, torch.full_like(bg, gap), bg)
    obs = inp["obs"].to(F64)
    y, x = torch.meshgrid(torch.arange(cam.height, device=DEV), torch.arange(cam.width, device=DEV), indexing="ij")
    base = _terms(_pad(bgz[None], w), obs[None], x, y, cam, lik, settings)
    mesh = inp["lattices"][slot]
    x0, y0, cw, ch = _crop_boxes(mesh, poses, cam, w + 1)
    if float(cw) * ch * poses.shape[0] > limit:
        return None
    total = [torch.zeros(poses.shape[0], dtype=F64, device=DEV) for _ in base]
    per = max(1, int(6e6 // (cw * ch)))
    pad_bg = _pad(bgz, w)
    ey, ex = torch.meshgrid(torch.arange(-w, ch + w, device=DEV), torch.arange(-w, cw + w, device=DEV), indexing="ij")
    for i in range(0, poses.shape[0], per):
        px = x0[i:i + per, None, None] + ex  # the crop and its margin, which may leave the image
        py = y0[i:i + per, None, None] + ey
        rx, ry = _rays(cam, px, py)
        B = px.shape[0]
        z = _cast(mesh, poses[i:i + per], rx.reshape(B, -1), ry.reshape(B, -1), far).reshape(px.shape)
        b = pad_bg[py + w, px + w]
        outside = (px < 0) | (py < 0) | (px >= cam.width) | (py >= cam.height)
        z = torch.where((z < far) & ~outside & ~(b <= z), z, b)
        inner = (slice(None), slice(w, w + ch), slice(w, w + cw))
        gx, gy = px[inner], py[inner]
        for g, l in enumerate(_terms(z, obs[gy, gx], gx, gy, cam, lik, settings)):
            total[g][i:i + per] = base[g].sum() + (l - base[g][0][gy, gx]).sum((1, 2))
    return total


def _exact_images(case, seed, limit=1.2e9):
    """(inputs, depth images [n, H, W]) of a render or camera case, or None."""
    if float(case["n"]) * case["width"] * case["height"] > limit:
        return None
    inp = _inputs(case, seed)
    sc, cam, poses = inp["scene"], inp["scene"].camera, inp["poses"]
    far = float(np.float32(cam.far))
    n = poses.shape[0]
    if case["kind"] == "camera":
        out = torch.empty((n, cam.height, cam.width), dtype=F64, device=DEV)
        world = torch.as_tensor(sc.poses.astype(np.float64), device=DEV)
        rx, ry = _image_rays(cam)
        per = max(1, int(6e6 // rx.numel()))
        for i in range(0, n, per):
            P = poses[i:i + per].to(F64)
            R = rx.expand(P.shape[0], -1).contiguous(), ry.expand(P.shape[0], -1).contiguous()
            z = torch.full_like(R[0], far)
            for k, m in enumerate(inp["lattices"]):
                z = torch.minimum(z, _cast(m, P @ world[k], *R, far))
            out[i:i + per] = z.reshape(-1, cam.height, cam.width)
        return inp, out
    bg = _fixed_depth(sc, inp["lattices"], sc.poses, inp["slot"])
    out = bg.repeat(n, 1, 1)
    mesh = inp["lattices"][inp["slot"]]
    x0, y0, cw, ch = _crop_boxes(mesh, poses, cam, 1)
    per = max(1, int(6e6 // (cw * ch)))
    ey, ex = torch.meshgrid(torch.arange(ch, device=DEV), torch.arange(cw, device=DEV), indexing="ij")
    for i in range(0, n, per):
        px, py = x0[i:i + per, None, None] + ex, y0[i:i + per, None, None] + ey
        rx, ry = _rays(cam, px, py)
        B = px.shape[0]
        z = _cast(mesh, poses[i:i + per], rx.reshape(B, -1), ry.reshape(B, -1), far).reshape(px.shape)
        k = torch.arange(i, i + B, device=DEV)[:, None, None]
        out[k, py, px] = torch.minimum(out[k, py, px], z)
    return inp, out


def _exact_full(inp, depth, lik):
    """Sum of l_i of whole images [n, H, W]."""
    cam = inp["scene"].camera
    w = lik["half_window"]
    obs = inp["obs"].to(F64)
    y, x = torch.meshgrid(torch.arange(cam.height, device=DEV), torch.arange(cam.width, device=DEV), indexing="ij")
    per = max(1, int(6e6 // (cam.height * cam.width)))
    return torch.cat([_terms(_pad(depth[i:i + per], w), obs[None].expand(min(per, depth.shape[0] - i), -1, -1), x, y, cam,
                             lik)[0].sum((1, 2)) for i in range(0, depth.shape[0], per)])


def _exact_grad(case, seed):
    """Log-likelihood of the smooth likelihood and its derivatives with respect to the left se(3)
    perturbation (visibility fixed, rendered points sliding along their rays on their faces),
    sigma and p_out."""
    if float(case["n"]) * case["width"] * case["height"] > 1e8:
        return None
    inp = _inputs(case, seed)
    sc, slot, cam = inp["scene"], inp["slot"], inp["scene"].camera
    lik, far, w = _lik(case), float(np.float32(cam.far)), case["half_window"]
    s, p, V, K = _constants(lik, cam)
    bg = _fixed_depth(sc, inp["lattices"], sc.poses, slot)
    obs = inp["obs"].to(F64)
    ok = (obs > 0) & torch.isfinite(obs)
    rx, ry = _image_rays(cam)
    ix, iy = rx.reshape(cam.height, cam.width), ry.reshape(cam.height, cam.width)
    H, W = cam.height, cam.width
    gauss = (2 * math.pi * s * s) ** -1.5
    out = [[], [], [], []]
    for i in range(0, case["n"], 64):
        P = inp["poses"][i:i + 64].to(F64)
        B = P.shape[0]
        z, axis = _cast(inp["lattices"][slot], P, rx.expand(B, -1).contiguous(), ry.expand(B, -1).contiguous(), far, True)
        z, axis = z.reshape(B, H, W), axis.reshape(B, H, W)
        mine = (axis >= 0) & (z < bg)
        z = torch.where(mine, z, bg)
        zp = _pad(z, w)
        jx, jy = _pad(ix, w), _pad(iy, w)
        E, D = torch.zeros_like(z), torch.zeros_like(z)
        shifts = [(dy, dx) for dy in range(2 * w + 1) for dx in range(2 * w + 1)]

        def cut(a, dy, dx):
            return a[..., dy:dy + H, dx:dx + W]

        for dy, dx in shifts:
            q = cut(zp, dy, dx)
            d2 = (obs * ix - q * cut(jx, dy, dx)) ** 2 + (obs * iy - q * cut(jy, dy, dx)) ** 2 + (obs - q) ** 2
            e = torch.nan_to_num(torch.exp(-d2 / (2 * s * s)))
            E += e
            D += e * torch.nan_to_num(d2 / (s * s) - 3.0)
        dens = p / V + (1 - p) / K * gauss * E
        out[0].append(torch.where(ok, torch.log(dens), torch.zeros_like(dens)).sum((1, 2)))
        out[2].append(torch.where(ok, (1 - p) / K * gauss * D / (s * dens), torch.zeros_like(dens)).sum((1, 2)))
        out[3].append(torch.where(ok, (1 / V - gauss * E / K) / dens, torch.zeros_like(dens)).sum((1, 2)))
        weight = _pad(torch.where(ok, (1 - p) / K / dens, torch.zeros_like(dens)), w)
        op = _pad(obs, w)
        g = torch.zeros_like(z)
        for dy, dx in shifts:  # observed pixels whose window holds this rendered point
            qi, ax, ay, wt = (cut(a, dy, dx) for a in (op, jx, jy, weight))
            ex, ey, ez = qi * ax - z * ix, qi * ay - z * iy, qi - z
            t = wt * gauss * torch.exp(-(ex ** 2 + ey ** 2 + ez ** 2) / (2 * s * s)) * (ex * ix + ey * iy + ez) / (s * s)
            g += torch.where(torch.isfinite(t), t, torch.zeros_like(t))
        N = _inv3(P[:, :3, :3]).transpose(1, 2)  # columns: the face normals of the three axes
        nrm = N.transpose(1, 2)[torch.arange(B, device=DEV)[:, None, None], axis.long().clamp(min=0)]
        q = torch.stack([z * ix, z * iy, z], -1)
        nr = nrm[..., 0] * ix + nrm[..., 1] * iy + nrm[..., 2]
        dz = torch.cat([nrm, torch.linalg.cross(q, nrm)], -1) / nr[..., None]
        dz = torch.where(mine[..., None] & torch.isfinite(dz), dz, torch.zeros_like(dz))
        out[1].append((g[..., None] * dz).sum((1, 2)))
    return tuple(torch.cat(o) for o in out)


def exact(case, seed):
    kind = case["kind"]
    if kind == "resample":
        ll = torch.as_tensor(synth.random_ll(np.random.default_rng([9, int(seed)]), case["n"])).to(F64)
        return torch.logsumexp(ll, 0, keepdim=True), None, None
    if kind == "score":
        got = _exact_scores(case, seed)
        return None if got is None else got[0]
    if kind == "multi":
        parts = [_exact_scores(c, seed + 1000003 * k, limit=1e8) for k, c in enumerate(_multi_cases(case))]
        return [None if p is None else p[0] for p in parts]
    if kind == "noise":
        radii, pouts = _noise(case)
        settings = [(r, p) for r in radii for p in pouts]
        got = _exact_scores(case, seed, settings)
        if got is None:
            return None
        ll = torch.stack(got, 1)
        return ll, torch.logsumexp(ll - math.log(len(settings)), 1)
    if kind == "render":
        got = _exact_images(case, seed)
        return None if got is None else (got[1], None)
    if kind in ("materialised", "camera"):
        got = _exact_images(case, seed)
        return None if got is None else (got[1], _exact_full(*got, _lik(case)))
    if kind == "grad":
        return _exact_grad(case, seed)
    return None  # a whole enumeration: its draws depend on every score's last bit
