"""The scan of the tiles' pair counts where a block takes several rounds (more
than 2^18 sub-buckets), with split lists in several rounds: pairs and ranges
bit-exact, and an overflow's true pair count."""
import ctypes

import pytest

import synth

from gpu_common import compare_integers, require_gpu, run_gpu

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width,height", ((2048, 2048), (2064, 2064), (4096, 4080)))   # 1, 2 and 4 rounds
def test_many_tiles(width, height):
    require_gpu()
    from paper_2412_04459_gb300 import DeviceScene, Frame, _native as N
    scene = synth.dense_scene(5, seed=6)
    cam = synth.orbit_camera(3, width, height, distance=20.0 * width / 2048)
    fr, out, ins = run_gpu(scene, cam)
    lens = ins["ranges"][:, 1].astype(int) - ins["ranges"][:, 0]
    assert (lens > 1024).sum() > 4
    compare_integers(scene, cam, ins)
    small = Frame(DeviceScene.from_host(scene), cam, pair_capacity=1000)
    small.preprocess()
    n = ctypes.c_int64(0)
    assert N.lib().svr_bin_sort(N.ref(small.frame), N.ref(n), None) == N.SVR_ERR_CAPACITY
    assert n.value == ins["n_pairs"]
