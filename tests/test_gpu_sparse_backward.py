"""Backward where most voxels fall between the pixels' centres: only the
accumulators of voxels that a pixel can hit are cleared and read.  Batches
around the view loops' step of four, voxel counts around a word of 32, a
workspace full of NaN before the call, against the oracle and against the views
one by one."""
import numpy as np
import pytest

import oracle
import synth

from gpu_common import compare_grads, compare_reordered, oracle_grads, require_gpu

pytestmark = pytest.mark.gpu


def scene_of(n):
    return synth.scenes.subscene(synth.dense_scene(5, seed=8), np.random.default_rng(n).permutation(32768)[:n])


def gradients(dev, cams, ups, batched):
    """d_grid, d_sh, priorities; the workspace holds NaN before, and the call is
    made twice (the second with the accumulators of the first behind it)."""
    import torch
    from paper_2412_04459_gb300 import Frame
    fr = Frame(dev, cams if batched else cams[0], K=1)
    fr._alloc()
    fr.ws.fill_(0xFF)
    out = fr.render()
    g = [torch.cat([torch.from_numpy(np.ascontiguousarray(u[k])).float().reshape(-1) for u in ups]).cuda()
         for k in range(3)]
    for scale in (3.0, 1.0):
        prio = torch.zeros(dev.n_vox, device="cuda")
        d_grid, d_sh = fr.backward_ex(*[scale * x for x in g], out, priority=prio)
    return [x.double().cpu().numpy() for x in (d_grid, d_sh, prio)]


@pytest.mark.parametrize("n", (31, 33, 1000, 32768))
def test_one_view(n):
    require_gpu()
    from paper_2412_04459_gb300 import DeviceScene
    scene, cam = scene_of(n), synth.orbit_camera(3, 48, 40, distance=3.5)
    keep = oracle.render(scene, cam, K=1)["near_stop"] == 0
    up = [x * keep for x in synth.upstream_grads(1, 40, 48)]
    d_grid, d_sh, _ = gradients(DeviceScene.from_host(scene), [cam], [up], False)
    og, osh, mag = oracle_grads(scene, cam, *up, K=1)
    compare_grads(d_grid, og, name="grid", mag=(mag["grid"], mag["grid_seg"]))
    compare_grads(d_sh, osh, name="sh", mag=(mag["sh"], mag["sh_seg"]))


@pytest.mark.parametrize("views", (1, 3, 4, 5, 9))
def test_batches(views):
    require_gpu()
    from paper_2412_04459_gb300 import DeviceScene
    dev = DeviceScene.from_host(scene_of(20011))
    cams = [synth.orbit_camera(3 + v, 40 + 8 * v, 40, distance=3.5) for v in range(views)]
    ups = [synth.upstream_grads(v, 40, 40 + 8 * v) for v in range(views)]
    batch = gradients(dev, cams, ups, True)
    one_by_one = [sum(x) for x in zip(*(gradients(dev, [c], [u], False) for c, u in zip(cams, ups)))]
    for name, a, b in zip(("grid", "sh", "priority"), batch, one_by_one):
        assert np.abs(b).max() > 0
        compare_reordered(a, b, name)
