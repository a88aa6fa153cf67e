"""The work whose speed is looked after: calls through the public entry points
of paper_1903_11785_gb300.fvv on synthetic captures.

A capture is a ring of calibrated pinhole cameras around a box with players in
it (each a union of six ellipsoids), their exact silhouettes with 0.1% of the
pixels flipped, and colour images.  Four kinds of call are measured:

* ``frames``  silhouettes in, coloured mesh out: upload, reconstruct, colour and
              read the result, one frame at a time or a batch of frames in one
              call, from device memory or from pinned host memory;
* ``view``    a novel view of a reconstructed frame (the viewer moved);
* ``colour``  a reconstructed batch coloured again for other viewpoints;
* ``label``   the allocation-free labelling of an occupancy grid.

Launch shapes are the library's defaults: nothing here is tuned to a case.
"""
import ctypes
import math
import types

import numpy as np
import torch

from paper_1903_11785_gb300 import fvv

FLIPS = 1e-3            # silhouette pixels flipped, as by a segmentation's noise
# a player 1.8 m tall: ellipsoid centres and semi-axes (x to the side, z up)
BODY = (((-0.09, 0.0, 0.45), (0.08, 0.08, 0.45)), ((0.09, 0.0, 0.45), (0.08, 0.08, 0.45)),
        ((0.0, 0.0, 1.20), (0.20, 0.13, 0.35)), ((0.0, 0.0, 1.66), (0.10, 0.10, 0.12)),
        ((-0.25, 0.0, 1.20), (0.06, 0.06, 0.33)), ((0.25, 0.0, 1.20), (0.06, 0.06, 0.33)))
# counts of a reconstruction that its definition fixes (lookups_* say what a kernel chose to read)
COUNTS = ("flags", "n_components", "n_rois", "n_coarse_on", "n_fine_words", "n_verts", "n_tris", "tests_coarse",
          "tests_fine", "tests_bisect")

# Capture set-ups: the shapes of the repository's synthetic scenes.
TINY = dict(cams=8, width=640, height=360, focal=500.0, ring_x=6.0, ring_y=6.0, lift_lo=3.0, lift_hi=3.0, vol_x=4.0,
            vol_y=4.0, vol_z=2.5, coarse=0.05, fine=0.01, steps=8, players=1)
HD720 = dict(cams=8, width=1280, height=720, focal=1000.0, ring_x=8.0, ring_y=8.0, lift_lo=4.0, lift_hi=4.0,
             vol_x=8.0, vol_y=8.0, vol_z=2.5, coarse=0.05, fine=0.01, steps=8, players=3)
COURT = dict(cams=16, width=1920, height=1080, focal=1800.0, ring_x=30.0, ring_y=20.0, lift_lo=6.0, lift_hi=10.0,
             vol_x=20.0, vol_y=11.0, vol_z=4.0, coarse=0.05, fine=0.01, steps=10, players=12)
COURT_4K = dict(cams=10, width=3840, height=2160, focal=3600.0, ring_x=30.0, ring_y=20.0, lift_lo=6.0, lift_hi=10.0,
                vol_x=18.0, vol_y=18.0, vol_z=9.0, coarse=0.05, fine=0.02, steps=10, players=12)
MAT_4K = dict(cams=12, width=3840, height=2160, focal=3600.0, ring_x=14.0, ring_y=14.0, lift_lo=6.0, lift_hi=6.0,
              vol_x=12.0, vol_y=12.0, vol_z=3.0, coarse=0.04, fine=0.005, steps=12, players=3)
MAT = dict(cams=16, width=1920, height=1080, focal=1800.0, ring_x=14.0, ring_y=14.0, lift_lo=6.0, lift_hi=6.0,
           vol_x=5.0, vol_y=6.0, vol_z=2.1, coarse=0.08, fine=0.04, steps=10, players=3)
OPTIONS = dict(kind="frames", frames=1, width_step=0, height_step=0, abstain=False, pixel_walk=False, graphs=False,
               source="device")


def listed():
    def case(name, setup, **more):
        return {"name": name, **OPTIONS, **setup, **more}

    return [
        # the smallest capture, one frame at a time: launches and latency
        case("one small frame", TINY),
        # a live preview: one 720p frame at a time on a stream of its own, launch sequence replayed as a graph
        case("720p frame, graph", HD720, graphs=True),
        # the match capture, one frame at a time: latency at full size
        case("court frame", COURT),
        # a serving request: masks and colour images pinned on the host and read in place, mesh back to the host
        case("court frame, host", COURT, source="host"),
        # the same capture offline: 64 frames of a recording in one call
        case("court batch 64", COURT, frames=64),
        # the paper's match shape: ten 4K cameras, a volume that they do not all see (abstaining cameras)
        case("4K court batch 4", COURT_4K, frames=4, abstain=True),
        # grappling at 5 mm: the largest single frame
        case("4K mat frame", MAT_4K),
        # the paper's judo shape with its own surface rule (Eqs. (2)-(3)), a few frames at a time
        case("mat batch 8, pixel walk", MAT, frames=8, pixel_walk=True),
        # a mixed rig: seven cameras, none alike, sizes that no power of two divides
        case("mixed rig frame", HD720, cams=7, width=1277, height=723, width_step=54, height_step=31, fine=0.013,
             steps=7, players=2),
        # the viewer moves: a full-HD novel view of a reconstructed frame, zoomed in on the play
        case("novel view", COURT, kind="view", view_width=1920, view_height=1080, zoom=3.0),
        # the viewer of a paused clip moves: 8 meshes coloured again
        case("recolour 8", COURT, kind="colour", frames=8),
        # labelling inside a host program that may not allocate: the match capture's grid
        {"name": "label grid", "kind": "label", "nx": 400, "ny": 220, "nz": 80, "players": 13, "noise": 3e-4},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choices(("frames", "view", "colour", "label"), (12, 3, 2, 3))[0]
    if kind == "label":
        nx, ny, nz = int(_log(rng, 50, 420)), int(_log(rng, 50, 300)), int(_log(rng, 20, 180))
        nz = min(nz, 8388608 // (nx * ny))
        # either players and stray voxels, or a dense random grid (one large component and its islands)
        noise = rng.choice((min(3e-4, 3000.0 / (nx * ny * nz)), round(rng.uniform(0.22, 0.5), 3)))
        return {"kind": "label", "nx": nx, "ny": ny, "nz": nz, "players": rng.randint(1, 14), "noise": noise}
    vx, vy, vz = round(_log(rng, 4, 20), 1), round(_log(rng, 4, 14), 1), round(rng.uniform(2.2, 6.0), 1)
    width = int(_log(rng, 480, 3840))
    if rng.random() < 0.5:
        width -= width % 32
    height = max(270, int(width * rng.choice((9 / 16, 3 / 4, 0.5625 + 0.1 * rng.random()))))
    cams = rng.choice((6, 7, 8, 9, 10, 12, 14, 16, 16, 20))
    mixed = rng.random() < 0.25
    away = rng.uniform(1.4, 2.0)
    fine = round(_log(rng, 0.008, 0.04), 4)
    players = min(rng.randint(1, 12), max(1, int(vx * vy / 6)))
    # frames: as many as stay well below the largest listed case in pixels, mesh and coarse voxels
    coarse = round(rng.uniform(max(0.04, 1.5 * fine), max(0.08, 2.5 * fine)), 3)
    most = min(6.0e8 / (cams * width * height), 250.0 / (players * (0.01 / fine) ** 2),
               1.5e8 / (vx * vy * vz / coarse ** 3))
    frames = max(1, min(int(_log(rng, 1, 40)), int(most)))
    lift = round(rng.uniform(0.25, 0.45) * away * max(vx, vy) / 2 + 1.5, 1)
    case = dict(OPTIONS, kind=kind, frames=frames, cams=cams, width=width, height=height,
                width_step=rng.randint(1, 20) if mixed else 0, height_step=rng.randint(1, 10) if mixed else 0,
                focal=round(0.85 * width * min(1.0, 0.6 * away), 1), ring_x=round(away * max(vx, 4.0) / 1.2, 1),
                ring_y=round(away * max(vy, 4.0) / 1.1, 1), lift_lo=lift, lift_hi=lift + 1.0, vol_x=vx, vol_y=vy,
                vol_z=vz, coarse=coarse, fine=fine, steps=rng.randint(0, 12), players=players,
                abstain=rng.random() < 0.3, pixel_walk=rng.random() < 0.25, graphs=rng.random() < 0.3)
    if kind == "frames":
        case["source"] = "host" if rng.random() < 0.2 and frames * cams * width * height < 7e7 else "device"
    else:
        case["frames"] = 1 if kind == "view" else min(frames, 12)
        if kind == "view":
            case.update(view_width=int(_log(rng, 320, 3840)), view_height=int(_log(rng, 240, 2160)),
                        zoom=round(_log(rng, 0.8, 6.0), 2))
    return case


# ------------------------------------------------------------------ the capture

def _look_at(C, target, f, W, H, turn):
    fwd = target - C
    fwd = fwd / np.linalg.norm(fwd)
    right = np.cross(fwd, (0.0, 0.0, 1.0))
    right /= np.linalg.norm(right)
    R = np.stack([right, np.cross(fwd, right), fwd])
    a, b, c = turn
    Rz = np.array([[math.cos(a), -math.sin(a), 0], [math.sin(a), math.cos(a), 0], [0, 0, 1]])
    Ry = np.array([[math.cos(b), 0, math.sin(b)], [0, 1, 0], [-math.sin(b), 0, math.cos(b)]])
    Rx = np.array([[1, 0, 0], [0, math.cos(c), -math.sin(c)], [0, math.sin(c), math.cos(c)]])
    R = Rz @ Ry @ Rx @ R
    K = np.array([[f, 0, W / 2.0], [0, f, H / 2.0], [0, 0, 1.0]])
    return K @ np.concatenate([R, -R @ C[:, None]], axis=1)


def _setup(case, rng):
    """The calibrated cameras and reconstruction parameters of a capture."""
    n = case["cams"]
    W = [case["width"] - k * case["width_step"] for k in range(n)]
    H = [case["height"] - k * case["height_step"] for k in range(n)]
    P, C = [], []
    for k in range(n):
        a = 2 * math.pi * (k + rng.uniform(0.3, 0.7)) / n
        c = np.array([case["ring_x"] * math.cos(a), case["ring_y"] * math.sin(a),
                      rng.uniform(case["lift_lo"], case["lift_hi"] + 1e-9)])
        P.append(_look_at(c, np.array([0.0, 0.0, 0.9]), case["focal"] * W[k] / case["width"], W[k], H[k],
                          rng.uniform(-0.03, 0.03, 3)))
        C.append(c)
    return types.SimpleNamespace(
        P=np.stack(P).astype(np.float32), centre=np.stack(C).astype(np.float32), P64=np.stack(P), C64=np.stack(C),
        width=np.asarray(W, np.int32), height=np.asarray(H, np.int32), n_cams=n,
        vol_min=(-case["vol_x"] / 2, -case["vol_y"] / 2, 0.0),
        vol_max=(case["vol_x"] / 2, case["vol_y"] / 2, case["vol_z"]), coarse_m=case["coarse"], fine_m=case["fine"],
        bisect_steps=case["steps"], t_np=8, t_nb=2 ** 31 - 1, t_v=0.5,
        oob_policy=fvv.FVV_OOB_ABSTAIN if case["abstain"] else fvv.FVV_OOB_STRICT,
        surface_rule=fvv.FVV_SURFACE_LAMBDA if case["pixel_walk"] else fvv.FVV_SURFACE_BISECT)


def _players(case, rng):
    """(frames, players, 6) ellipsoid centres and rotated semi-axes, the players on smooth paths."""
    K, F = case["players"], case["frames"]
    hx, hy = 0.42 * case["vol_x"], 0.42 * case["vol_y"]
    base = []
    while len(base) < K:
        for _ in range(300):
            p = np.array([rng.uniform(-hx, hx), rng.uniform(-hy, hy)])
            if all(np.linalg.norm(p - q) >= 0.9 for q in base):
                break
        base.append(p)
    c0, ax = np.array([b[0] for b in BODY]), np.array([b[1] for b in BODY])
    centres, axes = np.zeros((F, K, 6, 3)), np.zeros((F, K, 6, 3, 3))
    for k in range(K):
        s, yaw = rng.uniform(1.7, 1.95) / 1.8, rng.uniform(0, 2 * math.pi)
        amp, om = rng.uniform(0.05, 0.4, 2), rng.uniform(0.5, 3.0, 2)
        for f in range(F):
            t = f / 30.0
            y = yaw + 0.4 * math.sin(om[0] * t)
            R = np.array([[math.cos(y), -math.sin(y), 0], [math.sin(y), math.cos(y), 0], [0, 0, 1]])
            at = np.clip(base[k] + amp * np.sin(om * t), (-hx, -hy), (hx, hy))
            centres[f, k] = np.array([at[0], at[1], 0.0]) + s * c0 @ R.T
            axes[f, k] = s * R[None] * ax[:, None, :]
    return centres, axes


def _ellipses(P, centres, axes):
    """Image ellipses of ellipsoids: d^T inv(S) d <= 1 around c, for every camera."""
    T = np.zeros(centres.shape[:-1] + (4, 4))
    T[..., :3, :3], T[..., :3, 3], T[..., 3, 3] = axes, centres, 1.0
    Q = T @ np.diag([1.0, 1.0, 1.0, -1.0]) @ np.swapaxes(T, -1, -2)
    D = np.einsum("nij,...jk,nlk->n...il", P, Q, P)
    D = D / D[..., 2:, 2:]
    c = D[..., :2, 2]
    return c, c[..., :, None] * c[..., None, :] - D[..., :2, :2]


def _masks(rig, centres, axes, gen):
    """(per-camera (H, W) uint8 masks of one frame) on the GPU."""
    c, S = _ellipses(rig.P64, centres, axes)                      # (N, K, 6, ...)
    half = np.sqrt(np.stack([S[..., 0, 0], S[..., 1, 1]], -1))
    lo = np.floor((c - half).min(axis=2)).astype(np.int64)        # (N, K, 2)
    size = (np.ceil((c + half).max(axis=2)).astype(np.int64) - lo + 1).max(axis=(0, 1))
    N, K = lo.shape[:2]
    dev = lambda x, t=torch.float32: torch.as_tensor(np.ascontiguousarray(x), dtype=t, device="cuda")  # noqa: E731
    M = np.linalg.inv(S)
    inv, mid = dev(M), dev(c - lo[:, :, None, :] - 0.5)           # ellipse centres relative to the crop's first pixel
    xs = torch.arange(int(size[0]), device="cuda", dtype=torch.float32)
    ys = torch.arange(int(size[1]), device="cuda", dtype=torch.float32)
    inside = torch.zeros((N, K, len(ys), len(xs)), dtype=torch.bool, device="cuda")
    for e in range(6):
        dx = xs[None, None, None, :] - mid[:, :, e, 0, None, None]
        dy = ys[None, None, :, None] - mid[:, :, e, 1, None, None]
        a, b, d = (inv[:, :, e, i, j, None, None] for i, j in ((0, 0), (0, 1), (1, 1)))
        inside |= (a * dx + 2 * b * dy) * dx + d * dy * dy <= 1.0
    W, H = dev(rig.width, torch.int64), dev(rig.height, torch.int64)
    sizes = [(int(h), int(w)) for h, w in zip(rig.height, rig.width)]
    starts = np.concatenate([[0], np.cumsum([-(-h * w // 256) * 256 for h, w in sizes])])
    px = dev(lo[..., 0], torch.int64)[:, :, None, None] + torch.arange(len(xs), device="cuda")[None, None, None, :]
    py = dev(lo[..., 1], torch.int64)[:, :, None, None] + torch.arange(len(ys), device="cuda")[None, None, :, None]
    inside &= (px >= 0) & (py >= 0) & (px < W[:, None, None, None]) & (py < H[:, None, None, None])
    at = dev(starts[:-1], torch.int64)[:, None, None, None] + py * W[:, None, None, None] + px
    flat = (torch.rand(int(starts[-1]), generator=gen, device="cuda") < FLIPS)
    full = torch.zeros_like(flat)
    full[at[inside]] = True
    flat ^= full
    flat = flat.view(torch.uint8)
    return [flat[s:s + h * w].view(h, w) for s, (h, w) in zip(starts, sizes)]


def _capacity(case):
    """Slot capacities a program sizes for its scene: 3 m^3 of fine grid and 80,000 vertices a player at 1 cm."""
    words = int((case["players"] + 2) * 3.0 / case["fine"] ** 3 / 32 * 1.4) + (1 << 16)
    verts = int((case["players"] + 1) * 80000 * (0.01 / case["fine"]) ** 2) + 8192
    return dict(max_fine_words=min(words, 1 << 23), max_verts=verts, max_tris=int(2.2 * verts))


def _capture(case, seed):
    rng = np.random.default_rng([1903, 11785, int(seed)])
    gen = torch.Generator(device="cuda").manual_seed(int(seed) + 1)
    s = types.SimpleNamespace(case=case, setup=_setup(case, rng), slots=list(range(case["frames"])))
    centres, axes = _players(case, rng)
    s.masks = [_masks(s.setup, centres[f], axes[f], gen) for f in range(case["frames"])]
    s.rgb = [[torch.randint(0, 256, m.shape + (3,), dtype=torch.uint8, device="cuda", generator=gen) for m in ms]
             for ms in s.masks]
    cam = int(rng.integers(s.setup.n_cams))
    path = [0.6 * s.setup.C64[(cam + f) % s.setup.n_cams] + 0.4 * s.setup.C64[(cam + f + 1) % s.setup.n_cams]
            for f in range(case["frames"])]
    s.viewpoints = (np.stack(path) + (0.0, 0.0, 0.5)).astype(np.float32)
    caps = _capacity(case)
    s.rig = fvv.Rig(s.setup, max_slots=case["frames"], host_staging=0, **caps)
    s.stream = None
    if case["graphs"]:
        s.stream = torch.cuda.Stream()
        s.rig.set_graphs(True)
    s.in_place = case["source"] == "host"
    if s.in_place:
        s.masks = [[m.cpu().pin_memory() for m in ms] for ms in s.masks]
        s.rgb = [[c.cpu().pin_memory() for c in cs] for cs in s.rgb]
    # the result buffers that a program keeps: (frames, capacity, ...), zero past each frame's mesh
    F, V, T = case["frames"], caps["max_verts"], caps["max_tris"]
    put = dict(device="cpu", pin_memory=True) if s.in_place else dict(device="cuda")
    s.out = {"verts": torch.zeros((F, V, 3), dtype=torch.float32, **put),
             "tris": torch.zeros((F, T, 3), dtype=torch.int32, **put),
             "rgb": torch.zeros((F, V, 3), dtype=torch.uint8, **put),
             "cam": torch.zeros((F, V), dtype=torch.int32, **put)}
    torch.cuda.synchronize()
    return s


def prepare(case, seed):
    if case["kind"] == "label":
        return _grid(case, seed)
    s = _capture(case, seed)
    if case["kind"] == "frames":
        s.each = [{k: v[f] for k, v in s.out.items()} for f in s.slots]
        return s
    s.rig.upload_silhouettes_batch(s.slots, s.masks, stream=s.stream)
    s.rig.reconstruct(s.slots, stream=s.stream)
    torch.cuda.synchronize()
    if case["kind"] == "colour":
        s.each = [{k: s.out[k][f] for k in ("rgb", "cam")} for f in s.slots]
        return s
    w, h = case["view_width"], case["view_height"]
    s.centre = s.viewpoints[0]
    s.P = _look_at(s.centre.astype(np.float64), np.array([0.0, 0.0, 0.9]), case["zoom"] * case["focal"] * w / case["width"], w,
                   h, (0.0, 0.0, 0.0)).astype(np.float32)
    return s


def run(state):
    s = state
    if isinstance(s, dict):
        return _label(s)
    rig, kind = s.rig, s.case["kind"]
    if kind == "view":
        key, rgb, cam = rig.render_view(0, s.rgb[0], s.P, s.centre, s.case["view_width"], s.case["view_height"],
                                        stream=s.stream)
        return {"key": key, "rgb": rgb, "cam": cam}
    if kind == "frames":
        rig.upload_silhouettes_batch(s.slots, s.masks, stream=s.stream, in_place=s.in_place)
        rig.reconstruct(s.slots, stream=s.stream)
    rig.colour(s.slots, s.rgb, s.viewpoints, stream=s.stream, in_place=s.in_place)
    counts = fvv.fvv_get_results_batch(rig.ptr, s.slots, s.each, stream=s.stream)
    counts = np.array([[c[k] for k in COUNTS] for c in counts])
    if kind == "colour":
        return {"rgb": s.out["rgb"], "cam": s.out["cam"]}
    return {"counts": counts, **s.out}


# ------------------------------------------------------------------ labelling

def _grid(case, seed):
    rng = np.random.default_rng([785, int(seed)])
    gen = torch.Generator(device="cuda").manual_seed(int(seed) + 2)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    nxw = (nx + 31) // 32
    occ = torch.rand((nz, ny, nxw * 32), generator=gen, device="cuda") < case["noise"]
    z, y, x = (torch.arange(n, device="cuda", dtype=torch.float32) for n in (nz, ny, nxw * 32))
    for _ in range(case["players"]):                              # a standing player at 5 cm a voxel
        cx, cy, cz = rng.uniform(0, nx), rng.uniform(0, ny), 18.0
        occ |= ((x / 6 - cx / 6) ** 2)[None, None, :] + ((y / 5 - cy / 5) ** 2)[None, :, None] + \
            ((z / 18 - cz / 18) ** 2)[:, None, None] <= 1.0
    bit = torch.ones(32, dtype=torch.int64, device="cuda") << torch.arange(32, device="cuda")
    occ = occ & (torch.arange(nxw * 32, device="cuda") < nx)
    words = (occ.view(nz, ny, nxw, 32).to(torch.int64) * bit).sum(-1)
    words = torch.where(words >= 1 << 31, words - (1 << 32), words).to(torch.int32).contiguous()
    return {"words": words, "dims": (nx, ny, nz), "labels": torch.zeros((nz, ny, nx), dtype=torch.int32, device="cuda"),
            "counts": torch.zeros(3, dtype=torch.int32, device="cuda")}


def _label(s):
    nx, ny, nz = s["dims"]
    ptr = lambda t: ctypes.c_void_p(t.data_ptr())  # noqa: E731
    status = fvv._lib.fvv_label_components_noalloc(
        ptr(s["words"]), nx, ny, nz, 8, 2 ** 31 - 1, ptr(s["labels"]), ptr(s["counts"]),
        ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
    if status != fvv.FVV_OK:
        raise RuntimeError(f"fvv_label_components_noalloc: status {status}")
    return {"labels": s["labels"], "counts": s["counts"]}


# ------------------------------------------------------------------ what a pass cannot do without

def work(case):
    """Each input byte the rule needs read once, each output written once; the
    floating-point operations of the method's own steps (a camera test is 22:
    three rows of a projection, two divisions, two floors).  Mesh sizes are
    those of players of 1.8 m: about 30,000 vertices and 60,000 triangles each
    at 1 cm."""
    if case["kind"] == "label":
        nvox = case["nx"] * case["ny"] * case["nz"]
        return {"bytes": nvox / 8 + 4 * nvox, "flops": 0}
    F, N = case["frames"], case["cams"]
    pixels = sum((case["width"] - k * case["width_step"]) * (case["height"] - k * case["height_step"])
                 for k in range(N))
    verts = 30000.0 * case["players"] * (0.01 / case["fine"]) ** 2
    tris = 2 * verts
    if case["kind"] == "view":
        view = case["view_width"] * case["view_height"]
        return {"bytes": 48 * tris + 15 * view, "flops": 68 * tris}
    colour = verts * (12 + 4 + 3 + 3 + 4), verts * 30              # position, depth and colour in; colour, camera out
    if case["kind"] == "colour":
        return {"bytes": F * colour[0], "flops": F * colour[1]}
    voxels = case["vol_x"] * case["vol_y"] * case["vol_z"] / case["coarse"] ** 3
    flops = 22 * voxels + 22 * verts * (1 + case["steps"]) + 20 * verts * N + colour[1]
    return {"bytes": F * (pixels + 12 * verts + 12 * tris + colour[0]), "flops": F * flops}


def exact(case, seed):
    """No value: every output is a discrete function of the silhouettes
    (indices, bytes, cameras, labels; a vertex is a dyadic point of a grid
    edge that a sequence of binary32 in/out decisions picks).  In 64 bits a few
    samples of a frame fall on the other side of a pixel's border, and the mesh
    then has other vertices in other places of the list."""
    return None
