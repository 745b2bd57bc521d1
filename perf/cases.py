"""The work that a user of this rasterizer has it do, as measurable cases.

A case is a dict of plain values; prepare() makes what a program holds before
the call (a scene on the GPU, cameras, a frame or a captured step), run() is
one pass through the public entry points, work() the bytes and operations that
the pass cannot do without, exact() the same outputs in 64 bits by plain torch
(every pixel ray against every voxel).

Scenes are adaptive octrees around noisy sphere shells (thin dense surfaces in
a sparse coarse background, the structure of a trained scene), random octrees
and dense grids, all generated on the GPU from the seed.
"""
import dataclasses
import math

import numpy as np
import torch

from paper_2412_04459_gb300 import raster, train
from paper_2412_04459_gb300.autotune import BatchedRenderer
from paper_2412_04459_gb300.raster import DeviceScene, Frame, rasterize, supersampled_camera

T_STOP = 1e-4
DEV = "cuda"


# ------------------------------------------------------------------- the cases

def listed():
    return [
        # the smallest call: a preview of a handful of voxels through the
        # differentiable entry point, inference only; launches and host work
        dict(name="tiny_view", kind="rasterize", scene="octree", voxels=64, width=48, height=40, K=3, grad=False),
        # one optimisation step of a coarse dense grid, as at the start of a
        # training run (forward and backward through autograd)
        dict(name="dense_grid_step", kind="rasterize", scene="dense", voxels=32768, width=128, height=128, K=1,
             grad=True),
        # a small scene at an odd image size over a white background, K = 2
        dict(name="ragged_step", kind="rasterize", scene="shell", voxels=24576, width=333, height=217, K=2,
             grad=True, bg=1.0),
        # a walk-through camera in the middle of the scene with a wide field
        # of view: voxels across the image plane are listed in every tile
        dict(name="inside_view", kind="view", scene="shell", voxels=98304, width=640, height=480, K=1, inside=True),
        # a low-resolution preview of a large scene while navigating: forward
        # only, one sample per voxel, many voxels per tile
        dict(name="preview", kind="view", scene="shells3", voxels=2 << 20, width=320, height=210, K=1),
        # the 1M-voxel forward and backward step, K = 3
        dict(name="step_1m", kind="step", scene="shell", voxels=1 << 20, width=1280, height=840, K=3),
        # a high-quality frame: rendered at 1.1 times its size, averaged down
        dict(name="view_antialiased", kind="view_ss", scene="shells3", voxels=2 << 20, width=1752, height=1168, K=3,
             h_ss=1.1),
        # every extra output: normals, pruning and subdivision statistics
        dict(name="extras_step", kind="extras", scene="shell", voxels=1 << 18, width=640, height=480, K=2),
        # a whole training step of the 1M-voxel scene: render, losses,
        # backward, Adam (captured forward and backward)
        dict(name="train_1m", kind="train", scene="shell", voxels=1 << 20, width=1280, height=840, K=3, views=1,
             h_ss=0.0, stats=False),
        # a training step over a few views with supersampling and the
        # statistics that the next octree edit needs
        dict(name="train_views", kind="train", scene="shell", voxels=1 << 18, width=504, height=378, K=1, views=4,
             h_ss=1.1, stats=True),
        # mixed-size views of one scene in one captured batch
        dict(name="batch_mixed", kind="batch", scene="shell", voxels=1 << 20, width=1280, height=840, K=3, views=16,
             mixed=True, tile=16),
        # the largest: 8 views of 2560 x 1440 on 8M voxels, forward and backward
        dict(name="batch_large", kind="batch", scene="shells3", voxels=8_000_000, width=2560, height=1440, K=3,
             views=8, mixed=False, tile=16),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges: image edges from 40 to 2560 pixels,
    64 to 4M voxels, K 1..3, 1 to 12 views."""
    kind = rng.choice(["rasterize", "view", "step", "view_ss", "extras", "train", "batch"])
    scene = rng.choice(["shell", "shell", "shells3", "octree", "dense"])
    lo, hi = dict(octree=(64, 4096), dense=(512, 32768), shell=(8192, 4 << 20), shells3=(65536, 4 << 20))[scene]
    voxels = _log_int(rng, lo, hi)
    if scene == "dense":
        voxels = 8 ** max(3, min(4 if kind == "rasterize" else 5, round(math.log(voxels, 8))))
    # coarse scenes are the start of a training run: small images
    height = _log_int(rng, 40, dict(dense=360, octree=480).get(scene, 1440))
    width = max(40, min(2560, int(height * rng.uniform(0.75, 1.9))))
    if scene.startswith("shell"):
        voxels = max(8192, min(voxels, 32 * width * height))
    case = dict(kind=kind, scene=scene, voxels=voxels, width=width, height=height, K=rng.randint(1, 3))
    if kind == "rasterize":   # the autograd call allocates its workspace: small scenes and images
        case["voxels"] = min(voxels, 16384)
        case["height"] = min(height, 400)
        case["width"] = min(width, 560)
        case["grad"] = rng.random() < 0.7
        case["bg"] = float(rng.choice([0.0, 1.0]))
    elif kind == "view":
        if voxels <= 131072 and width * height <= 1 << 20:
            case["inside"] = rng.random() < 0.3
    elif kind == "view_ss":
        case["h_ss"] = rng.choice([1.1, 1.5])
    elif kind == "train":
        case["views"] = rng.randint(1, 4)
        case["h_ss"] = rng.choice([0.0, 1.1, 1.5])
        case["stats"] = rng.random() < 0.5
    elif kind == "batch":
        case["views"] = rng.randint(2, 12)
        case["mixed"] = rng.random() < 0.5
        case["tile"] = rng.choice([8, 16, 16, 32])
    # at most half the largest listed case's view-pixels, a quarter of its
    # view-voxels (a larger tile takes more workspace per pair)
    while case.get("views", 1) > 1 and (case["views"] * case["width"] * case["height"] > 14_000_000 or
                                        case["views"] * case["voxels"] > 16_000_000):
        case["views"] -= 1
    return case


# ---------------------------------------------------------------------- inputs

@dataclasses.dataclass(frozen=True)
class Camera:
    """OpenCV pinhole; w2c = [R | t] float32 [3, 4]."""
    fx: np.float32
    fy: np.float32
    cx: np.float32
    cy: np.float32
    w2c: np.ndarray
    width: int
    height: int


def _look_at(eye, target, width, height, fov_x_deg):
    z = target - eye
    z = z / np.linalg.norm(z)
    up = np.array([0.0, 1.0, 0.0]) if abs(z[1]) < 0.99 else np.array([0.0, 0.0, 1.0])
    x = np.cross(z, up)
    x = x / np.linalg.norm(x)
    R = np.stack([x, np.cross(z, x), z])
    w2c = np.concatenate([R, (-R @ eye)[:, None]], axis=1).astype(np.float32)
    f = np.float32(0.5 * width / math.tan(math.radians(fov_x_deg) * 0.5))
    return Camera(f, f, np.float32(0.5 * width), np.float32(0.5 * height), w2c, int(width), int(height))


def _cameras(case, seed):
    rng = np.random.default_rng([int(seed), 17])
    centre = np.array([0.5, 0.5, 0.5])
    sizes = [(case["width"], case["height"])] * case.get("views", 1)
    if case.get("mixed"):
        scale = [(1, 2), (1, 1), (3, 2)]   # 640 x 420, 1280 x 840, 1920 x 1260 around 1280 x 840
        sizes = [(max(8, w * scale[i % 3][0] // scale[i % 3][1]), max(8, h * scale[i % 3][0] // scale[i % 3][1]))
                 for i, (w, h) in enumerate(sizes)]
    cams = []
    for w, h in sizes:
        d = rng.normal(size=3)
        d = d / np.linalg.norm(d)
        if case.get("inside"):
            eye = centre + 0.05 * rng.uniform(-1, 1, size=3)
            cams.append(_look_at(eye, eye + d, w, h, 80.0))
        else:
            cams.append(_look_at(centre + 2.5 * d, centre, w, h, 50.0))
    return cams


def _gen(seed, salt):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 8 + salt)
    return g


_BITS = [(c >> 2 & 1, c >> 1 & 1, c & 1) for c in range(8)]


def _split_cells(ijk):
    return (ijk[:, None, :] * 2 + torch.tensor(_BITS, device=DEV)[None]).reshape(-1, 3)


class _Shells:
    """Noisy sphere shells: distance of points to the nearest one."""

    def __init__(self, kind, gen):
        if kind == "shells3":
            self.c = [(0.47, 0.5, 0.52), (0.53, 0.48, 0.5), (0.5, 0.52, 0.47)]
            self.r, self.band = [0.25, 0.33, 0.41], 0.01
        else:
            self.c, self.r, self.band = [(0.5, 0.5, 0.5)], [0.4], 0.02
        self.noise = [[2.0 * torch.rand(1, 1, n + 1, n + 1, n + 1, device=DEV, generator=gen) - 1.0
                       for n in (4, 8, 16)] for _ in self.r]

    def distance(self, p):
        best = None
        at = (2.0 * p - 1.0).view(1, -1, 1, 1, 3)
        for c, r, tables in zip(self.c, self.r, self.noise):
            n = sum(w * torch.nn.functional.grid_sample(t, at, align_corners=True).reshape(-1)
                    for t, w in zip(tables, (4 / 7, 2 / 7, 1 / 7)))
            d = ((p - torch.tensor(c, device=DEV)).norm(dim=1) - (r + 0.05 * n)).abs()
            best = d if best is None else torch.minimum(best, d)
        return best


def _leaves(case, gen, shells):
    """Leaf cells (level, ijk) of an octree with about case["voxels"] leaves."""
    target, kind = case["voxels"], case["scene"]
    if kind == "dense":
        lvl = max(1, round(math.log(target, 8)))
        n = 1 << lvl
        ax = torch.arange(n, device=DEV)
        ijk = torch.stack(torch.meshgrid(ax, ax, ax, indexing="ij"), -1).reshape(-1, 3)
        return torch.full((len(ijk),), lvl, device=DEV), ijk
    if kind == "octree":
        lvl, p = 1, 0.5
        ijk = torch.tensor(_BITS, device=DEV)
    else:
        lvl, p = 4, 0.58 if kind == "shell" else 0.51
        ax = torch.arange(16, device=DEV)
        ijk = torch.stack(torch.meshgrid(ax, ax, ax, indexing="ij"), -1).reshape(-1, 3)
    levels, cells, done = [], [], 0
    while True:
        u = torch.rand(len(ijk), device=DEV, generator=gen)
        if shells is not None:
            size = 1.0 / (1 << lvl)
            near = shells.distance((ijk.float() + 0.5) * size) <= shells.band + size * (math.sqrt(3.0) / 2)
            u = torch.where(near, u, torch.full_like(u, 2.0))
        go = u < p
        # split no more cells than the target allows: the leaf count so far,
        # plus 7 more per split cell
        room = max(0, (target - done - len(ijk)) // 7)
        if room > 0 and not bool(go.any()):
            go[u.argmin()] = True
        n_go = int(go.sum())
        last = n_go >= room or lvl >= 14
        if n_go > room:
            keep = torch.argsort(u)[:room]
            go = torch.zeros_like(go)
            go[keep] = True
        levels.append(torch.full((len(ijk) - int(go.sum()),), lvl, device=DEV))
        cells.append(ijk[~go])
        done += len(cells[-1])
        ijk = _split_cells(ijk[go])
        lvl += 1
        if last:
            levels.append(torch.full((len(ijk),), lvl, device=DEV))
            cells.append(ijk)
            return torch.cat(levels), torch.cat(cells)


def _scene(case, seed):
    gen = _gen(seed, 1)
    shells = _Shells(case["scene"], gen) if case["scene"].startswith("shell") else None
    level, ijk = _leaves(case, gen, shells)
    perm = torch.randperm(len(level), device=DEV, generator=gen)   # voxels are stored in no particular order
    level, ijk = level[perm], ijk[perm]
    corner = ijk[:, None, :] + torch.tensor(_BITS, device=DEV)[None]
    key = (level[:, None] << 51) | (corner[..., 0] << 34) | (corner[..., 1] << 17) | corner[..., 2]
    points, corner_idx = torch.unique(key.reshape(-1), return_inverse=True)
    if shells is not None:
        grid = torch.empty(len(points), device=DEV)
        for a in range(0, len(points), 1 << 24):
            k = points[a:a + (1 << 24)]
            p = torch.stack([(k >> s) & 0x1FFFF for s in (34, 17, 0)], -1).float() / (2.0 ** (k >> 51))[:, None]
            near = shells.distance(p) <= shells.band
            val = 2.0 + torch.randn(len(k), device=DEV, generator=gen)
            grid[a:a + (1 << 24)] = torch.where(near, val, torch.full_like(val, -4.0))
    else:
        grid = torch.randn(len(points), device=DEV, generator=gen)
    if case["scene"] != "dense":
        # the parameter array keeps room for the points that octree edits add
        room = torch.zeros(3 * case["voxels"] + 256, device=DEV)
        room[:len(grid)] = grid
        grid = room
    sh = 0.3 * torch.randn(len(level), 48, device=DEV, generator=gen)
    centre = ((ijk.double() + 0.5) / (2.0 ** level.double())[:, None]).float()
    return DeviceScene(centre.contiguous(), level.to(torch.uint8), corner_idx.view(-1, 8).to(torch.int32).contiguous(),
                       grid, sh, (0.5, 0.5, 0.5), 1.0, int(level.max()))


def _upstream(case, seed, *shapes):
    gen = _gen(seed, 2)
    return [torch.randn(*s, device=DEV, generator=gen) for s in shapes]


def prepare(case, seed):
    scene = _scene(case, seed)
    cams = _cameras(case, seed)
    cam, K, kind = cams[0], case["K"], case["kind"]
    H, W = cam.height, cam.width
    st = dict(case=case, scene=scene, cam=cam, kind=kind)
    if kind == "rasterize":
        st["bg"] = (case.get("bg", 0.0),) * 3
        if case["grad"]:
            st["grid"] = scene.grid.clone().requires_grad_(True)
            st["sh"] = scene.sh.clone().requires_grad_(True)
            st["g"] = _upstream(case, seed, (3, H, W), (H, W), (H, W))
    elif kind in ("view", "step"):
        st["frame"] = Frame(scene, cam, K=K, t_stop=T_STOP)
        if kind == "step":
            st["frame"].render()    # sizes the workspace; the steps then read nothing back
            st["g"] = _upstream(case, seed, (3, H, W), (H, W), (H, W))
    elif kind == "view_ss":
        st["frame"] = Frame(scene, supersampled_camera(cam, case["h_ss"]), K=K, t_stop=T_STOP)
    elif kind == "extras":
        st["frame"] = Frame(scene, cam, K=K, t_stop=T_STOP)
        st["g"] = _upstream(case, seed, (3, H, W), (H, W), (H, W), (3, H, W))
    elif kind == "train":
        gen = _gen(seed, 3)
        targets = [torch.rand(3, c.height, c.width, device=DEV, generator=gen) for c in cams]
        step = train.TrainStep(scene, cams, targets, K=K, t_stop=T_STOP, h_ss=case["h_ss"] or None,
                               stats=case["stats"])
        # a step in the middle of a run: Adam's second moments are those of
        # gradients like this step's
        step.forward_backward()
        for g, v in ((step.d_grid, step.v_grid), (step.d_sh, step.v_sh)):
            v.copy_(g * g + (g * g).mean())
        step.n_steps = 500
        if case["stats"]:
            step.max_weight.zero_()
            step.priority.zero_()
        st["step"] = step.capture()
        if case["stats"]:
            step.max_weight.zero_()
            step.priority.zero_()
    else:
        r = BatchedRenderer(scene, cams, K=K, t_stop=T_STOP, tile=case["tile"], partitions=1)
        for buf, g in zip(r.grads, _upstream(case, seed, *[(b.numel(),) for b in r.grads])):
            buf.copy_(g)
        st["batch"] = r.capture()
    return st


# ------------------------------------------------------------------- one pass

def run(st):
    case, scene, cam, kind = st["case"], st["scene"], st["cam"], st["kind"]
    K = case["K"]
    if kind == "rasterize":
        if not case["grad"]:
            with torch.no_grad():
                return rasterize(scene.grid, scene.sh, scene, cam, K=K, t_stop=T_STOP, bg=st["bg"])
        images = rasterize(st["grid"], st["sh"], scene, cam, K=K, t_stop=T_STOP, bg=st["bg"])
        d_grid, d_sh = torch.autograd.grad(images, (st["grid"], st["sh"]), st["g"])
        return [x.detach() for x in images] + [d_grid, d_sh]
    if kind == "view":
        out = st["frame"].render()
        return [out["rgb"], out["depth"], out["alpha"]]
    if kind == "step":
        # a training loop's call: no pair count is read back
        out = st["frame"].render(sync=False)
        d_grid, d_sh = st["frame"].backward(*st["g"], out)
        return [out["rgb"], out["depth"], out["alpha"], d_grid, d_sh]
    if kind == "view_ss":
        out = st["frame"].render()
        return [raster.downsample(out[k], cam.height, cam.width) for k in ("rgb", "depth", "alpha")]
    if kind == "extras":
        fr = st["frame"]
        max_weight = torch.zeros(scene.n_vox, device=DEV)
        priority = torch.zeros(scene.n_vox, device=DEV)
        fr.preprocess()
        fr.bin_sort()
        out = fr.forward_ex(normal=True, max_weight=max_weight)
        g_rgb, g_depth, g_alpha, g_normal = st["g"]
        d_grid, d_sh = fr.backward_ex(g_rgb, g_depth, g_alpha, out, g_normal=g_normal, priority=priority)
        return [out["rgb"], out["depth"], out["alpha"], out["normal"], max_weight, priority, d_grid, d_sh]
    if kind == "train":
        step = st["step"]
        loss = step.step()
        res = [loss, step.out["rgb"], step.d_grid, step.d_sh, scene.grid, scene.sh]
        return res + ([step.max_weight, step.priority] if case["stats"] else [])
    r = st["batch"]
    r.step()
    return [r.out["rgb"], r.out["depth"], r.out["alpha"], r.d_grid, r.d_sh]


# ----------------------------------------------------------------------- work

def work(case):
    """Each input read once and each output written once (float32); the
    operations of the composited samples at 6 voxels per pixel (background
    included), K samples each, about 33 operations a sample forward and twice
    that backward."""
    n, K, kind, views = case["voxels"], case["K"], case["kind"], case.get("views", 1)
    ss = case.get("h_ss") or 1.0
    px = views * case["width"] * case["height"]
    points = 3 * n if case["scene"] != "dense" else 1.1 * n
    back = kind in ("step", "extras", "train", "batch") or (kind == "rasterize" and case["grad"])
    scene = n * (12 + 1 + 32 + 192) + 4 * points
    nbytes = scene + px * 4 * 5
    flops = px * ss * ss * 6 * (30 + 33 * K)
    if back:
        nbytes += px * 4 * 5 + 4 * points + 192 * n
        flops *= 3
    if kind == "extras":
        nbytes += px * 4 * 6 + n * 8
    if kind == "train":
        nbytes += px * 4 * 3 + 28 * (points + 48 * n) + (n * 8 if case["stats"] else 0)
    return {"bytes": float(nbytes), "flops": float(flops)}


# ---------------------------------------------------------------------- exact

EXACT_MOST = 9e10          # ray-voxel tests of one case
EXACT_PIXELS = 400_000     # and pixels (the hits are held at once)


def exact(case, seed):
    """run()'s outputs in 64 bits: every pixel ray against every voxel (Sec.
    A.2), hits sorted by entry distance, composited front to back; gradients
    by torch's autograd through the same expressions."""
    kind = case["kind"]
    if kind in ("train", "batch"):
        return None
    ss = case.get("h_ss") or 1.0
    pixels = case["width"] * case["height"] * ss * ss
    if pixels * case["voxels"] > EXACT_MOST or pixels > EXACT_PIXELS:
        return None
    scene = _scene(case, seed)
    cam = _cameras(case, seed)[0]
    H, W = cam.height, cam.width
    if kind == "view_ss":
        cam_ss = _scaled(cam, case["h_ss"])
        img = _render64(scene, cam_ss, case["K"], 0.0)
        A, B = _area(H, cam_ss.height), _area(W, cam_ss.width)
        return [A @ x @ B.T for x in img[:3]]
    if kind == "view" or (kind == "rasterize" and not case["grad"]):
        return _render64(scene, cam, case["K"], case.get("bg", 0.0))[:3]
    normal = kind == "extras"
    shapes = [(3, H, W), (H, W), (H, W)] + ([(3, H, W)] if normal else [])
    g = [x.double() for x in _upstream(case, seed, *shapes)]
    img, max_weight, d_grid, d_sh = _render64(scene, cam, case["K"], case.get("bg", 0.0), g, normal)
    return img + ([max_weight, None] if normal else []) + [d_grid, d_sh]


def _scaled(cam, h_ss):
    Ws, Hs = int(round(h_ss * cam.width)), int(round(h_ss * cam.height))
    sx, sy = Ws / cam.width, Hs / cam.height
    return dataclasses.replace(cam, fx=np.float32(float(cam.fx) * sx), fy=np.float32(float(cam.fy) * sy),
                               cx=np.float32(float(cam.cx) * sx), cy=np.float32(float(cam.cy) * sy),
                               width=Ws, height=Hs)


def _area(n, n_ss):
    """Row x: overlap of source pixels with target pixel x's footprint, over its length."""
    X = torch.arange(n_ss, device=DEV, dtype=torch.float64)[None] * n
    x = torch.arange(n, device=DEV, dtype=torch.float64)[:, None] * n_ss
    return (torch.minimum(X + n, x + n_ss) - torch.maximum(X, x)).clamp(min=0) / n_ss


def _sh_colour(centre, origin, sh):
    d = centre - origin
    x, y, z = (d / d.norm(dim=1, keepdim=True)).unbind(1)
    pi = math.pi
    Y = [0.5 * math.sqrt(1 / pi) + 0 * x,
         math.sqrt(3 / (4 * pi)) * y, math.sqrt(3 / (4 * pi)) * z, math.sqrt(3 / (4 * pi)) * x,
         0.5 * math.sqrt(15 / pi) * x * y, 0.5 * math.sqrt(15 / pi) * y * z,
         0.25 * math.sqrt(5 / pi) * (3 * z * z - 1), 0.5 * math.sqrt(15 / pi) * x * z,
         0.25 * math.sqrt(15 / pi) * (x * x - y * y),
         0.25 * math.sqrt(35 / (2 * pi)) * y * (3 * x * x - y * y), 0.5 * math.sqrt(105 / pi) * x * y * z,
         0.25 * math.sqrt(21 / (2 * pi)) * y * (5 * z * z - 1), 0.25 * math.sqrt(7 / pi) * z * (5 * z * z - 3),
         0.25 * math.sqrt(21 / (2 * pi)) * x * (5 * z * z - 1), 0.25 * math.sqrt(105 / pi) * z * (x * x - y * y),
         0.25 * math.sqrt(35 / (2 * pi)) * x * (x * x - 3 * y * y)]
    return torch.relu((torch.stack(Y, 1)[:, :, None] * sh.view(-1, 16, 3)).sum(1))


def _hits64(lo, hi, origin, rays):
    """(pixel, voxel, a, b) of every valid ray-box segment (a <= b, a > 0)."""
    inv = 1.0 / (rays + 0.0)
    per = max(1, (1 << 26) // len(lo))
    found = []
    for p0 in range(0, len(rays), per):
        a = b = None
        for ax in range(3):
            i = inv[p0:p0 + per, ax, None]
            t0, t1 = (lo[:, ax] - origin[ax])[None] * i, (hi[:, ax] - origin[ax])[None] * i
            n, f = torch.minimum(t0, t1), torch.maximum(t0, t1)
            a, b = (n, f) if a is None else (torch.maximum(a, n), torch.minimum(b, f))
        pix, vox = ((a <= b) & (a > 0)).nonzero(as_tuple=True)
        found.append((pix + p0, vox, a[pix, vox], b[pix, vox]))
    return [torch.cat(x) for x in zip(*found)]


def _render64(scene, cam, K, bg, g=None, normal=False):
    w2c = torch.tensor(np.asarray(cam.w2c, np.float64), device=DEV)
    R, t = w2c[:, :3], w2c[:, 3]
    origin = -(R.T @ t)
    H, W = cam.height, cam.width
    y, x = torch.meshgrid(torch.arange(H, device=DEV, dtype=torch.float64) + 0.5,
                          torch.arange(W, device=DEV, dtype=torch.float64) + 0.5, indexing="ij")
    d = torch.stack([(x - float(cam.cx)) / float(cam.fx), (y - float(cam.cy)) / float(cam.fy), torch.ones_like(x)], -1)
    rays = (d.reshape(-1, 3) @ R).contiguous()
    centre = scene.centre.double()
    size = 2.0 ** -scene.level.double()
    lo = centre - 0.5 * size[:, None]
    behind = None
    for bits in _BITS:
        z = (lo + size[:, None] * torch.tensor(bits, device=DEV, dtype=torch.float64)) @ R[2] + t[2]
        behind = z <= 1e-3 if behind is None else behind & (z <= 1e-3)
    seen = (~behind).nonzero().reshape(-1)
    pix, vox, a, b = _hits64(lo[seen], (lo + size[:, None])[seen], origin, rays)
    vox = seen[vox]
    order = torch.argsort(a, stable=True)
    order = order[torch.argsort(pix[order], stable=True)]
    pix, vox, a, b = pix[order], vox[order], a[order], b[order]
    # place i of each hit among its pixel's: rows of a padded [pixels, most] table
    count = torch.bincount(pix, minlength=H * W)
    rank = torch.arange(len(pix), device=DEV) - (torch.cumsum(count, 0) - count)[pix]
    most = int(count.max()) if len(pix) else 1
    grid = scene.grid.double().requires_grad_(g is not None)
    sh = scene.sh.double().requires_grad_(g is not None)
    with torch.set_grad_enabled(g is not None):
        corners = grid[scene.corner_idx.long()[vox]]
        seg = (b - a)
        length = seg * rays[pix].norm(dim=1) / K
        e, ts = [], []
        for k in range(K):
            tk = a + (k + 0.5) * seg / K
            q = (origin + tk[:, None] * rays[pix] - lo[vox]) / size[vox][:, None]
            v = 0
            for c, bits in enumerate(_BITS):
                w = 1
                for ax in range(3):
                    w = w * (q[:, ax] if bits[ax] else 1 - q[:, ax])
                v = v + w * corners[:, c]
            sigma = torch.where(v > 1.1, v, 1.1 * torch.exp(torch.clamp(v, max=1.1) / 1.1 - 1))
            e.append(length * sigma)
            ts.append(tk)
        X = sum(e)
        alpha = -torch.expm1(-X)
        dloc, before = 0, 0
        for k in range(K):
            dloc = dloc + torch.exp(-before) * -torch.expm1(-e[k]) * ts[k] if k else -torch.expm1(-e[0]) * ts[0]
            before = before + e[k]
        table = torch.zeros(H * W, most, device=DEV, dtype=torch.float64).index_put((pix, rank), X)
        cum = torch.cumsum(table, 1)
        T = torch.exp(-(cum - table))[pix, rank]
        live = (T >= float(np.float32(T_STOP))).double()   # the walk stops after the voxel that leaves T < t_stop
        wgt = T * alpha * live
        colour = _sh_colour(centre, origin, sh)[vox]
        put = lambda v: torch.zeros(H * W, device=DEV, dtype=torch.float64).index_add(0, pix, v)  # noqa: E731
        T_final = torch.exp(-put(X * live))
        rgb = torch.stack([put(wgt * colour[:, c]) + T_final * bg for c in range(3)]).view(3, H, W)
        img = [rgb, put(T * dloc * live).view(H, W), (1 - T_final).view(H, W)]
        if normal:
            c = corners.view(-1, 2, 2, 2)
            n = 0.25 * torch.stack([(c[:, 1] - c[:, 0]).sum((1, 2)), (c[:, :, 1] - c[:, :, 0]).sum((1, 2)),
                                    (c[:, :, :, 1] - c[:, :, :, 0]).sum((1, 2))], 1)
            s = (n * n).sum(1)
            n = n * torch.where(s > 0, torch.rsqrt(torch.where(s > 0, s, torch.ones_like(s))), torch.zeros_like(s))[:, None]
            img.append(torch.stack([put(wgt * n[:, k]) for k in range(3)]).view(3, H, W))
    if g is None:
        return [v.detach() for v in img]
    d_grid, d_sh = torch.autograd.grad(img, (grid, sh), g)
    top = torch.zeros(scene.n_vox, device=DEV, dtype=torch.float64)
    top = top.scatter_reduce(0, vox, wgt.detach(), "amax")
    return [v.detach() for v in img], top, d_grid, d_sh
