"""Voxels over many tiles: a camera inside the scene, where voxels lie across
the camera plane and near it.  Their pairs (integers, bit-exact) and, since
the render narrows them to the pixels in front (and a tile's ray signs are
taken from its corners where those agree), the images, against the oracle."""
import numpy as np
import pytest

import oracle
import synth

from gpu_common import compare_images, compare_integers, require_gpu, run_gpu

pytestmark = pytest.mark.gpu

CASES = [
    # eye, target, fov, size, scene centre and size (a scene far from the
    # origin loses digits in the projection)
    ((0.52, 0.47, 0.44), (0.9, 0.6, 0.7), 80.0, (70, 50), (0.5, 0.5, 0.5), 1.0),
    ((0.53, 0.48, 0.46), (0.53, 0.48, 1.46), 100.0, (97, 41), (0.5, 0.5, 0.5), 1.0),   # along an axis
    ((0.1, 0.9, 0.3), (0.1, 0.2, 0.3), 60.0, (33, 129), (0.5, 0.5, 0.5), 1.0),
    ((40.3, -19.6, 7.1), (41.0, -20.4, 6.6), 90.0, (64, 64), (40.0, -20.0, 7.0), 2.0),
]


@pytest.mark.parametrize("case", range(len(CASES)))
@pytest.mark.parametrize("level", (2, 4))
def test_camera_inside(case, level):
    require_gpu()
    eye, target, fov, (w, h), centre, size = CASES[case]
    scene = synth.dense_scene(level, seed=case, center=centre, size=size)
    up = (0.0, 0.0, 1.0) if abs(target[0] - eye[0]) < 1e-3 and abs(target[2] - eye[2]) < 1e-3 else (0.0, 1.0, 0.0)
    cam = synth.look_at(eye, target, up, fov, w, h)
    fr, out, ins = run_gpu(scene, cam, K=2)
    compare_integers(scene, cam, ins)
    compare_images(out, oracle.render(scene, cam, K=2))


@pytest.mark.parametrize("size", ((1, 1), (16, 16), (17, 31), (130, 65)))
def test_tile_masks_on_the_axes(size):
    """Rays of every sign pattern around the optical axis: tiles whose corner
    pixels disagree are walked pixel by pixel.  (Integers only: the axis lies
    on voxel faces, where a ray's hits are not defined.)"""
    require_gpu()
    scene = synth.dense_scene(2, seed=1)
    for d in ((0.0, 0.0, -2.0), (0.01, 0.02, -2.0), (-2.0, 0.3, 0.0)):
        cam = synth.look_at(np.array([0.5, 0.5, 0.5]) + d, (0.5, 0.5, 0.5), (0.0, 1.0, 0.0), 50.0, *size)
        fr, out, ins = run_gpu(scene, cam)
        compare_integers(scene, cam, ins)
