"""Renders whose rays fit the resident lanes (the launch of Sec. 6 for previews, probes and thumbnails): they are dealt
out evenly, from one ray a warp to 32, instead of from the queue. A ray's result does not depend on who traces it, so
the images are equal bit for bit, whatever the grid; every ray is traced once."""
import numpy as np
import pytest

import paper_1704_02724_gb300 as cx
import synth
from gpu_util import config_canvas, render

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("block", [128, 256])
@pytest.mark.parametrize("traversal", [0, 1])
def test_rays_per_warp(block, traversal):
    cv = config_canvas(0)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    room = sms * (block // 32)                       # warps at one block an SM
    sizes = [(1, 1), (33, 2)]
    for take in (1, 2, 4, 8, 16, 32):                # tiles of 8 x 4 pixels: rays at and past room / 2 x take
        tiles = room // 2 * take // 32
        sizes += [(8 * tiles, 4), (8 * tiles + 8, 4)] if tiles else []
    sizes += [(8 * room, 4), (8 * room + 1, 4)]      # the last that fits one block an SM, and one more tile
    for w, h in sizes:
        cams = synth.cameras_array([synth.look_at_camera([0.1, 0.05, -0.9], [0.3, 0.1, 0.4], [0, 1, 0], 1.0, w, h, 0,
                                                         (0.1, 0.2, 0.3, 1.0))])
        ref, st = render(cv, cams, key="c0", block_threads=block, traversal=traversal, blocks_per_sm=1, refill=4)
        assert st["rays"] == w * h
        for kw in (dict(blocks_per_sm=1), dict(blocks_per_sm=4), dict(blocks_per_sm=4, per_view=1)):
            img, st = render(cv, cams, key="c0", block_threads=block, traversal=traversal, **kw)
            assert st["rays"] == w * h
            assert np.array_equal(img, ref), (w, h, kw)
