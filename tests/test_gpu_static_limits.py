"""Limits of the allocation-free forward render: calls between its limit and
what a workspace with the backward's buffers would leave are rendered, and
calls just beyond the limit are refused."""
import pytest

import synth

from gpu_common import IMG_TOL, require_gpu
from test_zz_no_alloc import _regular_render, _static_call

pytestmark = pytest.mark.gpu


# pairs 82,419 of 88,176 and 52,172 of 56,200 in the array; 88,960 of 87,812
@pytest.mark.parametrize("size,distance,fits", (((288, 216), 1.2, True), ((1280, 840), 14.0, True),
                                                ((320, 240), 1.2, False)))
def test_static_limit(size, distance, fits):
    require_gpu()
    from paper_2412_04459_gb300 import DeviceScene, _native as N
    dev = DeviceScene.from_host(synth.dense_scene(5, seed=1))
    cam = synth.orbit_camera(3, *size, distance=distance)
    rc, got, n_static = _static_call(dev, cam, 1, 1e-4, (0.0, 0.0, 0.0))
    ref, n_regular = _regular_render(dev, cam, 1, 1e-4, (0.0, 0.0, 0.0))
    assert n_static == n_regular
    assert rc == (0 if fits else N.SVR_ERR_CAPACITY)
    if fits:
        for k in ("rgb", "depth", "alpha", "T_final"):
            assert abs(got[k] - ref[k]).max() <= IMG_TOL, k
