"""Corner densities at the ends of the float range: points marked empty by the
lowest float, opaque by the highest, or by infinities, among ordinary ones.
Images and gradients against the oracle, which takes the same densities in 64
bits (those of the infinities as the lowest and highest float)."""
import numpy as np
import pytest

import oracle
import synth

from gpu_common import compare_images, oracle_grads, require_gpu

pytestmark = pytest.mark.gpu

MOST = float(np.finfo(np.float32).max)


@pytest.mark.parametrize("batched", (False, True))
@pytest.mark.parametrize("value", (-MOST, MOST, -np.inf, np.inf))
@pytest.mark.parametrize("level,share", ((1, 0.2), (3, 0.3), (3, 1.0)))
def test_ends_of_the_range(value, level, share, batched):
    require_gpu()
    import torch
    from paper_2412_04459_gb300 import DeviceScene, Frame

    def grid_fn(pos, rng):
        g = rng.normal(size=len(pos))
        return np.where(rng.random(len(pos)) < share, np.clip(value, -MOST, MOST), g)

    scene, cam = synth.dense_scene(level, seed=4, grid_fn=grid_fn), synth.orbit_camera(3, 64, 48, distance=1.9)
    ref = oracle.render(scene, cam, K=2)
    up = synth.upstream_grads(0, 48, 64)
    d_grid, d_sh, _ = oracle_grads(scene, cam, *up, K=2)
    scene.grid = np.where(np.abs(scene.grid) >= MOST, np.float32(value), scene.grid)
    fr = Frame(DeviceScene.from_host(scene), [cam] if batched else cam, K=2)
    out = fr.render()
    compare_images(fr.views(out)[0] if batched else out, ref)
    g = [torch.from_numpy(np.ascontiguousarray(x)).float().cuda() for x in up]
    got_grid, got_sh = fr.backward(*[x.reshape(-1) for x in g] if batched else g, out)
    for got, want in ((got_grid, d_grid), (got_sh, d_sh)):
        got, want = got.double().cpu().numpy().reshape(-1), np.asarray(want, np.float64).reshape(-1)
        # all opaque: terms that cancel to 0 in 64 bits leave roundings of each
        assert np.linalg.norm(got - want) <= 1e-3 * np.linalg.norm(want) + 1e-6 * np.sqrt(got.size)
