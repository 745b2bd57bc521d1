"""At the capacity that a frame takes by itself (four pairs per voxel and view) the
workspace is no larger than the buffers of the layout that had separate gradient
accumulators of 12 bytes per voxel and view: a scene that fitted still does."""
import pytest

import synth


def earlier_bytes(n, views, cap, tiles, tile):
    """Every buffer of that layout, on 256-byte boundaries."""
    B, VN = tile * tile // 32, views * n
    slots = 2 * cap // 1024 + 1
    seg = [8 * tiles, 4 * B * tiles, 4 * B * slots, 4 * B * slots * 14 * 32]
    sizes = [64, tiles * (1 + B), 8 * n, 8 * VN, 4 * VN, 4 * 17 * tiles, 64 * VN, 4 * ((8 * tiles + 255) // 256 + 1),
             8 * cap, 8 * cap, 4 * cap, 4 * cap, 8 * tiles, 12 * VN, 8 * VN, 8 * (tiles + slots), 8 * B * cap,
             4 * B * tiles, 4 * B * (cap + 32 * tiles), *seg]
    return sum((b + 255) // 256 * 256 for b in sizes)


@pytest.mark.parametrize("views", (1, 3, 8, 32))
@pytest.mark.parametrize("n,w,h", ((1 << 20, 1280, 840), (8_000_000, 2560, 1440), (2 << 20, 320, 210),
                                   (1 << 18, 640, 480)))
def test_no_larger_than_before(n, w, h, views):
    from paper_2412_04459_gb300 import build
    build.build()
    from paper_2412_04459_gb300.raster import workspace_size
    cam = synth.orbit_camera(3, w, h, distance=2.5)
    tiles = views * ((w + 15) // 16) * ((h + 15) // 16)
    cap = 4 * n * views
    if cap < 1 << 31:
        assert workspace_size(n, cap, [cam] * views, batched=True) <= earlier_bytes(n, views, cap, tiles, 16)
