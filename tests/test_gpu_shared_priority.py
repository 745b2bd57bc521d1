"""Backwards of two frames on two streams that add to one priority array (and
one density gradient): every term arrives."""
import numpy as np
import pytest

import synth

from gpu_common import require_gpu

pytestmark = pytest.mark.gpu

REPEATS = 8
# Sums of non-negative terms, a few hundred a voxel, in another order: relative
# error below 1,000 x 2^-24.  A lost update is at least 1 / (2 REPEATS) of the
# smaller frame's share of a voxel.
REL = 6e-5


def test_two_streams_add_to_one_priority():
    require_gpu()
    import torch
    from paper_2412_04459_gb300 import DeviceScene, Frame
    dev = DeviceScene.from_host(synth.dense_scene(6, seed=1))
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    work = []
    for i in range(2):
        cam = synth.orbit_camera(3 + i, 160, 120, distance=1.7)
        fr = Frame(dev, cam, K=1)
        out = fr.render()
        g = [torch.from_numpy(np.ascontiguousarray(x)).float().cuda() for x in synth.upstream_grads(i, 120, 160)]
        alone = torch.zeros(dev.n_vox, device="cuda")
        fr.backward_ex(*g, out, priority=alone)
        work.append((fr, out, g, alone, torch.empty(dev.n_vox, 48, device="cuda")))
    want = REPEATS * (work[0][3].double() + work[1][3].double())
    assert int(((work[0][3] > 0) & (work[1][3] > 0)).sum()) > 1000
    for _ in range(5):
        both, d_grid = torch.zeros(dev.n_vox, device="cuda"), torch.zeros_like(dev.grid)
        torch.cuda.synchronize()
        for _ in range(REPEATS):
            for s, (fr, out, g, _, d_sh) in zip(streams, work):
                with torch.cuda.stream(s):
                    fr.backward_ex(*g, out, priority=both, d_grid=d_grid, d_sh=d_sh)
        torch.cuda.synchronize()
        assert float(((both.double() - want).abs() - REL * want).max()) <= 0.0
