"""Frame.render with the pair count read back while the render runs, and the
memory that autograd calls leave behind."""
import gc

import numpy as np
import pytest

import synth

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu


def _scene_cam():
    return (synth.random_octree_scene(5, max_level=4, grid_fn=synth.normal_grid(0.5, 1.0)),
            synth.orbit_camera(3, 61, 47, distance=1.9))


def test_too_small_workspace_is_grown_and_the_view_redone():
    require_gpu()
    import torch
    from paper_2412_04459_gb300 import DeviceScene, Frame
    sc, cam = _scene_cam()
    dev = DeviceScene.from_host(sc)
    ref = Frame(dev, cam, K=2)
    want = ref.render()
    assert ref.n_pairs > 100
    fr = Frame(dev, cam, K=2, pair_capacity=100)
    for _ in range(2):   # grown on the first call, fits on the second
        out = fr.render()
        assert fr.n_pairs == ref.n_pairs <= fr.pair_capacity
        for k in want:
            assert torch.equal(out[k], want[k]), k


def test_invalid_voxel_raises():
    require_gpu()
    from paper_2412_04459_gb300 import DeviceScene, Frame, _native as N
    sc, cam = _scene_cam()
    sc.centre = np.array(sc.centre)
    sc.centre[0] += 0.4 * np.float32(2.0 ** -int(sc.level[0]))
    with pytest.raises(N.SvrError) as e:
        Frame(DeviceScene.from_host(sc), cam).render()
    assert e.value.code == N.SVR_ERR_INVALID


def test_autograd_calls_keep_no_memory():
    require_gpu()
    import torch
    from paper_2412_04459_gb300 import DeviceScene, rasterize
    sc, cam = _scene_cam()
    dev = DeviceScene.from_host(sc)
    grid, sh = dev.grid.clone().requires_grad_(True), dev.sh.clone().requires_grad_(True)

    def step():
        rgb, depth, alpha = rasterize(grid, sh, dev, cam, K=2)
        torch.autograd.grad(rgb.sum() + depth.sum() + alpha.sum(), (grid, sh))

    def held():
        gc.collect()
        torch.cuda.synchronize()
        return torch.cuda.memory_allocated()

    step()
    before = held()
    for _ in range(3):
        step()
    assert held() == before
