"""Addressing of the pools in the mixed traversal (Sec. 4.1.1: index-based pools): 32-bit byte offsets while records,
links and leaves each end below 4 GiB, 64-bit ones beyond. Depth-27 canvases of the device painter whose leaves end
just below and beyond that line, seen from inside the rooms (the deepest cells come last in the pools), against the
plain FP64 caster, which takes neither."""
import numpy as np
import pytest

import paper_1704_02724_gb300 as cx
import synth
from gpu_util import TOL, _uploaded

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_fine,small", [(150_000, True), (220_000, False)])
def test_offsets_near_4_gib(n_fine, small):
    D, E, c, r, q, _ = synth.config_stamps(3, n_fine=n_fine)
    _uploaded["key"] = None
    n_rec, n_leaf = cx.paint_spheres(D, E, c, r, q)
    assert (n_rec * 48 <= 2 ** 32 and n_leaf * 8 <= 2 ** 32) == small
    assert n_leaf * 8 > 3 * 2 ** 30          # byte offsets past 2^31 either way
    cams = synth.config_cameras(3, res_scale=64 / 2160)
    n = synth.total_pixels(cams)
    img = torch.empty((n, 4), device="cuda")
    ref = torch.empty((n, 4), device="cuda")
    cx.render(cams, ref, precision=cx.PREC_FP64)
    for kw in (dict(), dict(traversal=1), dict(count_reads=0), dict(precision=cx.PREC_FP64_LINKS)):
        cx.render(cams, img, **kw)
        assert float((img - ref).abs().max()) <= TOL, kw
    cx.release()                              # (tens of GB: back to the device)
