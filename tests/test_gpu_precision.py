"""Errors against the FP64 oracle, held to those of the kernels that evaluated
densities and gradients corner by corner with exp's fast form (figures taken on
these scenes): relative L2 errors of the images."""
import numpy as np
import pytest

import oracle
import synth

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu

SCENES = {
    "faint": lambda: synth.random_octree_scene(5, max_level=4, p_split=0.6, grid_fn=synth.normal_grid(-3.0, 0.5)),
    "mixed": lambda: synth.random_octree_scene(6, max_level=5, p_split=0.5, grid_fn=synth.normal_grid(0.0, 1.0)),
    "dense": lambda: synth.dense_scene(5, seed=2),
}
# the corner form's errors: depth
DEPTH = {("faint", 1): 5.47954e-06, ("faint", 2): 7.74346e-06, ("faint", 3): 1.04815e-05,
         ("mixed", 1): 5.14253e-07, ("mixed", 2): 7.31532e-07, ("mixed", 3): 9.51886e-07,
         ("dense", 1): 1.84280e-06, ("dense", 2): 2.90522e-06, ("dense", 3): 3.43589e-06}


def image_error(name, K, key):
    from paper_2412_04459_gb300 import DeviceScene, Frame
    scene, cam = SCENES[name](), synth.orbit_camera(3, 160, 120, distance=1.9)
    out = Frame(DeviceScene.from_host(scene), cam, K=K).render()
    ref = oracle.render(scene, cam, K=K)
    assert (ref["near_stop"] == 0).all()
    got = out[key].cpu().numpy().astype(np.float64)
    return np.linalg.norm(got - ref[key]) / np.linalg.norm(ref[key])


@pytest.mark.parametrize("name,K", sorted(DEPTH))
def test_depth(name, K):
    """P (1 - e) keeps the precision of 1 - e (as the difference of two rounded
    transmittances: 1.3 to 9 % more for two and three samples)."""
    require_gpu()
    assert image_error(name, K, "depth") <= 1.015 * DEPTH[name, K]


def test_small_shares_of_the_density_gradient():
    """A corner's gradient is its trilinear weight's share of the voxel's.  One
    voxel, one pixel, one sample near a corner: shares down to 1e-7 keep their
    relative precision.  The place q in the voxel is t r / size - c with |t r /
    size|, |c| <= 4, from operands of relative error below 2^-22: off by at
    most 3e-6 per axis, so a share with distance w to the far faces' weights 0 by
    3e-6 sum 1 / w, plus the products' roundings.  (Sums of polynomial
    coefficients taken to the corners are off by 2^-24 of the whole gradient.)"""
    require_gpu()
    import torch
    from paper_2412_04459_gb300 import DeviceScene, Frame
    scene = synth.scenes.subscene(synth.dense_scene(1, seed=3), np.array([7]))
    dev = DeviceScene.from_host(scene)
    lo, size = np.asarray(scene.centre[0], np.float64) - 0.25, 0.5
    rng = np.random.default_rng(11)
    smallest, done = 1.0, 0
    for _ in range(150):
        w = np.exp(rng.uniform(np.log(0.004), np.log(0.1), 3))
        corner = rng.integers(0, 2, 3)
        target = lo + size * np.where(corner, 1 - w, w)
        d = rng.normal(size=3)
        d /= np.linalg.norm(d)
        cam = synth.look_at(target - 1.2 * d, target, (0.0, 1.0, 0.0) if abs(d[1]) < 0.9 else (1.0, 0.0, 0.0), 40.0,
                            1, 1)
        w2c = np.asarray(cam.w2c, np.float64)
        origin, ray = -w2c[:, :3].T @ w2c[:, 3], w2c[2, :3]   # the pixel's centre is the principal point
        t = np.sort(np.stack([(lo - origin) / ray, (lo + size - origin) / ray]), 0)
        a, b = t[0].max(), t[1].min()
        q = (origin + 0.5 * (a + b) * ray - lo) / size
        near = np.minimum(q, 1 - q)
        if not (b - a > 1e-3 and near.max() < 0.2 and near.min() > 2e-3):
            continue
        fr = Frame(dev, cam, K=1)
        out = fr.render()
        d_grid, _ = fr.backward(torch.ones(3, 1, 1, device="cuda"), torch.zeros(1, 1, device="cuda"),
                                torch.ones(1, 1, device="cuda"), out)
        g = d_grid.double().cpu().numpy()[np.asarray(scene.corner_idx[0])]
        share = np.array([np.prod(np.where(np.array([c >> 2 & 1, c >> 1 & 1, c & 1]), q, 1 - q)) for c in range(8)])
        rel = np.abs(g / g.sum() / share - 1).max()
        assert rel <= 3e-6 * (1 / near).sum() + 1e-6, (rel, share.min())
        smallest, done = min(smallest, share.min()), done + 1
    assert done >= 10 and smallest < 1e-5


# the corner form's errors: alpha, one sample
ALPHA = {"mixed": 5.00171e-07, "dense": 1.91148e-06}


@pytest.mark.parametrize("name", sorted(ALPHA))
def test_alpha(name):
    """explin's exponent takes log2(e) as a factor of its own (folded into its
    two constants: 0.6 to 1 % more).  The forward is deterministic."""
    require_gpu()
    assert image_error(name, 1, "alpha") <= 1.004 * ALPHA[name]


def single_voxel(value):
    scene = synth.scenes.subscene(synth.dense_scene(1, seed=3, grid_fn=synth.constant_grid(value)), np.array([7]))
    centre = np.asarray(scene.centre[0], np.float64)
    cam = synth.look_at(centre + np.array([0.4, 0.3, -2.0]), centre, (0.0, 1.0, 0.0), 20.0, 24, 16)
    w2c = np.asarray(cam.w2c, np.float64)
    origin = -w2c[:, :3].T @ w2c[:, 3]
    x, y = np.meshgrid((np.arange(24) + 0.5 - float(cam.cx)) / float(cam.fx),
                       (np.arange(16) + 0.5 - float(cam.cy)) / float(cam.fy))
    rays = np.stack([x, y, np.ones_like(x)], -1) @ w2c[:, :3]
    t = np.sort(np.stack([(centre - 0.25 - origin) / rays, (centre + 0.25 - origin) / rays]), 0)
    length = np.maximum(t[1].min(-1) - t[0].max(-1), 0.0) * np.linalg.norm(rays, axis=-1)
    return scene, cam, length


TINY = 2.0 ** -149   # spacing of the subnormals


@pytest.mark.parametrize("K", (1, 2, 3))
@pytest.mark.parametrize("value", (-90.0, -97.0, -100.0, -104.0))
def test_densities_below_the_normal_range(value, K):
    """A voxel of density explin(v) < 2^-126 (v < -95.2) has a weight.  The
    exponent, about -140, is off by three roundings of 2^-18 each at most, and
    each of some ten subnormal products and sums by one spacing.  (Gradients
    that small are flushed by the global atomics in any case.)"""
    require_gpu()
    import torch
    from paper_2412_04459_gb300 import DeviceScene, Frame
    scene, cam, length = single_voxel(value)
    fr = Frame(DeviceScene.from_host(scene), cam, K=K)
    fr.preprocess()
    fr.bin_sort()
    weight = torch.zeros(1, device="cuda")
    fr.forward_ex(max_weight=weight)
    sigma = 1.1 * np.exp(value / 1.1 - 1.0)
    want = length.max() * sigma
    assert abs(float(weight) - want) <= 1e-4 * want + 10 * TINY


def test_transmittance_below_the_normal_range():
    """exp(-x) for optical depths from 87.3 (2^-126) to 103 (2^-149) is not
    flushed: relative error below that of x, 103 x 2^-21, plus one spacing."""
    require_gpu()
    from paper_2412_04459_gb300 import DeviceScene, Frame
    scene, cam, length = single_voxel(0.0)
    depth = 95.0 / length.max()
    scene, cam, length = single_voxel(float(np.float32(depth)))
    T = Frame(DeviceScene.from_host(scene), cam, K=1).render()["T_final"].double().cpu().numpy()
    want = np.exp(-length * float(np.float32(depth)))
    sel = (want < 2.0 ** -126) & (length > 0)
    assert sel.sum() > 20
    assert (np.abs(T - want)[sel] <= 1e-4 * want[sel] + 2 * TINY).all()
