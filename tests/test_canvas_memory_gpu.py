"""A canvas that replaces another is laid into its memory where it fits (canvases that grow, shrink, repeat, and are
uploaded, painted and appended to in turn): every one equals the same canvas made in fresh memory."""
import numpy as np
import pytest

import paper_1704_02724_gb300 as cx
import synth
from gpu_util import _uploaded

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _stamps(n):
    rng = np.random.default_rng(n)
    c = rng.uniform(-0.45, 0.45, (n, 3))
    r = np.exp(rng.uniform(np.log(0.02), np.log(0.1), n))
    return c, r, np.c_[rng.uniform(0, 1, (n, 3)), rng.uniform(0, 9, n)].astype(np.float32)


def _state(cams):
    out = torch.zeros((synth.total_pixels(cams), 4), device="cuda")
    cx.render(cams, out)
    nodes, leaves = cx.download_octree()
    host, dev = cx.octree_hash()
    assert host == dev
    return nodes, leaves, out.cpu().numpy()


@pytest.mark.parametrize("sizes", [(40, 40), (40, 80, 40), (200, 40, 41, 300), (1, 300, 1)])
def test_canvases_in_turn(sizes):
    cams = synth.config_cameras(0, res_scale=0.25)
    fresh = {}
    for n in set(sizes):
        cx.release()
        cx.paint_spheres(7, 1.0, *_stamps(n))
        fresh[n] = _state(cams)
        c, r, q = _stamps(5)
        cx.paint_append(c, r, q)
        fresh[n, 5] = _state(cams)
    cx.release()
    _uploaded["key"] = None
    for step, n in enumerate(sizes + sizes):
        if step % 2:
            cx.upload_octree(fresh[n][0], fresh[n][1], 7, 1.0)
        else:
            cx.paint_spheres(7, 1.0, *_stamps(n))
        for a, b in zip(_state(cams), fresh[n]):
            assert np.array_equal(a, b)
        if step % 2 == 0:
            cx.paint_append(*_stamps(5))
            for a, b in zip(_state(cams), fresh[n, 5]):
                assert np.array_equal(a, b)
