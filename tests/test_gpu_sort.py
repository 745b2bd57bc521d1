"""The per-tile sort at the edges of its length classes: lists around 32, 128
and every class boundary, around one and several chunks, with pairs that fit
one 64-bit word (level 10) and pairs that do not (level 15 with 2^16 voxels,
level 16 with 2^13, where the values break ties), against the oracle's emission
and np.lexsort order: bit-exact keys, values and ranges."""
import numpy as np
import pytest

import synth
from synth.scenes import Cells, make_scene

from gpu_common import compare_integers, require_gpu, run_gpu

pytestmark = pytest.mark.gpu

LENGTHS = (1, 2, 31, 32, 33, 127, 128, 129, 255, 256, 257, 511, 512, 513, 1023, 1024, 1025, 2047, 2048, 2049, 4095,
           4096, 4097, 8191, 8192, 8193, 12289, 16384, 16385, 40001)
# voxels that no view holds, so that a voxel id takes more bits
UNSEEN = {10: 0, 15: 1 << 16, 16: 1 << 13}


def lattice_scene(n, level, seed):
    """n distinct cells of one level around the scene centre (they share their
    top Morton bits, as the voxels of one surface crossing do), and UNSEEN
    cells far to the side."""
    rng = np.random.default_rng(seed)
    side, span = 1 << level, 64
    flat = rng.choice(span ** 3, size=n, replace=False)
    ijk = np.stack([flat // span ** 2, flat // span % span, flat % span], 1) + (side - span) // 2
    far = np.zeros((UNSEEN[level], 3), np.int64)
    far[:, 0] = side - 1
    ijk = np.concatenate([ijk, far]).astype(np.int64)
    cells = Cells(ijk, np.full(len(ijk), level, np.int64), (ijk + 0.5) / side, np.full(len(ijk), 1.0 / side))
    return make_scene(cells, lambda pos, r: r.normal(size=len(pos)), 0.3, rng)


@pytest.mark.parametrize("n", LENGTHS)
@pytest.mark.parametrize("level", sorted(UNSEEN))
def test_list_lengths(n, level):
    require_gpu()
    scene = lattice_scene(n, level, n + level)
    # a 16 x 16 image (one tile) over the cells, its rays of one sign pattern
    cam = synth.look_at((-1.2, -1.1, -1.4), (0.5, 0.5, 0.5), (0.0, 1.0, 0.0), 5.0, 16, 16)
    fr, out, ins = run_gpu(scene, cam)
    assert ins["n_pairs"] == n
    compare_integers(scene, cam, ins)


# eyes whose view holds the cells in its middle tile and not the far cells
EYES = {10: (-1.2, -1.1, -1.4), 15: (0.85, 0.2, 0.2)}


@pytest.mark.parametrize("n", (8193, 16385, 40001))
@pytest.mark.parametrize("level", sorted(EYES))
def test_long_list_among_many_tiles(n, level):
    """Images of more than 8192 tiles merge their long lists with smaller
    clusters."""
    require_gpu()
    scene = lattice_scene(n, level, n + level)
    # 91 x 91 tiles, the cells a few pixels wide
    cam = synth.look_at(EYES[level], (0.5, 0.5, 0.5), (0.0, 1.0, 0.0), 150.0, 1456, 1456)
    fr, out, ins = run_gpu(scene, cam)
    assert (ins["ranges"][:, 1].astype(np.int64) - ins["ranges"][:, 0]).max() == n
    compare_integers(scene, cam, ins)
