"""Pairs of one tile with equal keys, which the value orders: at max level 16
two sign patterns' rays can see mirrored cells in one order, and at any level
voxels may overlap (one given twice, or with its first child).  Pairs that do
not fit one 64-bit word, lists within one sorting group, of several chunks and
merged by clusters of eight and of two; keys that hold padded sign triples
below the sorted bits (level 14); tiles with several sign patterns.  Keys,
values and ranges bit-exact against the oracle's np.lexsort by (key, value)."""
import numpy as np
import pytest

import synth
from synth.scenes import Cells, make_scene

from gpu_common import compare_integers, require_gpu, run_gpu

pytestmark = pytest.mark.gpu

SPAN = 64


def scene_of(ijk, level, unseen, unseen_level, on_axis, seed):
    """The given cells, and `unseen` cells behind or far beside the camera that
    only raise the number of bits of a voxel id."""
    rng = np.random.default_rng(seed)
    far = np.zeros((unseen, 3), np.int64)
    far[:, 0] = 0 if on_axis else (1 << unseen_level) - 1
    ijk = np.concatenate([ijk, far]).astype(np.int64)
    level = np.concatenate([level, np.full(unseen, unseen_level)]).astype(np.int64)
    order = rng.permutation(len(ijk))   # ids in no particular order
    ijk, level = ijk[order], level[order]
    size = 0.5 ** level
    return make_scene(Cells(ijk, level, (ijk + 0.5) * size[:, None], size), lambda pos, r: r.normal(size=len(pos)), 0.3, rng)


def central(n, level, seed):
    """n distinct cells of the 64^3 around the lattice's middle."""
    flat = np.random.default_rng(seed).choice(SPAN ** 3, size=n, replace=False)
    return np.stack([flat // SPAN ** 2, flat // SPAN % SPAN, flat % SPAN], 1) + ((1 << level) - SPAN) // 2


def camera(tiles, on_axis):
    """One tile, or 91 x 91 with the cells in the middle one; along the x axis
    (the middle tile's rays have four sign patterns) or from a corner (one)."""
    eye = (0.3, 0.5, 0.5) if on_axis else (0.85, 0.2, 0.2)
    fov, edge = (5.0, 16) if tiles == 1 else (150.0, 1456)
    return synth.look_at(eye, (0.5, 0.5, 0.5), (0.0, 1.0, 0.0), fov, edge, edge)


def check(scene, cam, n_pairs, ties):
    fr, out, ins = run_gpu(scene, cam)
    compare_integers(scene, cam, ins)
    assert ins["n_pairs"] == n_pairs
    equal = int((np.diff(ins["keys"].astype(np.uint64)) == 0).sum())   # the oracle's keys, compared above
    assert (equal > 0) == ties


@pytest.mark.parametrize("tiles,cells", ((1, 16), (1, 100), (1, 1024), (1, 2046), (1, 2048), (1, 2050), (1, 6000),
                                         (8281, 2050), (8281, 6000)))
def test_mirrored_cells_at_level_16(tiles, cells):
    require_gpu()
    half = central(cells // 2, 16, cells)
    half = half[half[:, 1] < 1 << 15]
    mirror = half.copy()
    mirror[:, 1:] = (1 << 16) - 1 - mirror[:, 1:]
    ijk = np.concatenate([half, mirror])
    scene = scene_of(ijk, np.full(len(ijk), 16), 1 << 13, 16, True, cells)
    check(scene, camera(tiles, True), 4 * len(ijk), True)


@pytest.mark.parametrize("tiles,cells", ((1, 40), (1, 700), (1, 5000), (1, 9000), (1, 20000), (8281, 5000),
                                         (8281, 20000)))
def test_overlapping_voxels(tiles, cells):
    require_gpu()
    ijk = central(cells, 15, cells)
    parents = np.unique(ijk[ijk.sum(1) % 5 == 0] // 2, axis=0)
    ijk = np.concatenate([ijk, ijk[::3], 2 * parents])   # twice, and first children
    level = np.concatenate([np.full(len(ijk), 15), np.full(len(parents), 14)])
    scene = scene_of(np.concatenate([ijk, parents]), level, 1 << 16, 15, False, cells)
    check(scene, camera(tiles, False), len(level), True)


@pytest.mark.parametrize("tiles,cells", ((1, 75), (1, 2049), (1, 4097), (8281, 4097)))
def test_padded_triples_below_the_sorted_bits(tiles, cells):
    require_gpu()
    scene = scene_of(central(cells, 14, cells), np.full(cells, 14), 1 << 19, 14, True, cells)
    check(scene, camera(tiles, True), 4 * cells, False)
