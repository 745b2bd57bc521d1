"""Calls under a caller's default device: the first synchronised render of a
thread allocates its page-locked status words on the host."""
import threading

import pytest

import synth

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu


def test_render_with_cuda_as_default_device():
    require_gpu()
    import torch
    from paper_2412_04459_gb300 import DeviceScene, Frame, rasterize
    dev = DeviceScene.from_host(synth.dense_scene(3, seed=1))
    cam = synth.orbit_camera(3, 48, 40, distance=1.9)
    want = Frame(dev, cam).render()
    got, error = [], []

    def call():   # a thread of its own: nothing is allocated for it yet
        try:
            with torch.device("cuda"):
                got.append(Frame(dev, cam).render()["rgb"])
                got.append(rasterize(dev.grid, dev.sh, dev, cam)[0])
        except Exception as e:  # noqa: BLE001
            error.append(e)

    t = threading.Thread(target=call)
    t.start()
    t.join()
    assert not error, error
    torch.cuda.synchronize()
    for rgb in got:
        assert torch.equal(rgb, want["rgb"])
