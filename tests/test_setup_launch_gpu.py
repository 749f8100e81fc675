"""A render's set-up (Sec. 4.1.5: views and starting cells before the rays): up to 64 views travel as the arguments of
one launch, in two sizes of argument block; more views, and renders replayed from a graph, are staged in pinned memory.
Either way the rays get the same words, so the images are equal bit for bit."""
import numpy as np
import pytest

import paper_1704_02724_gb300 as cx
import synth
from gpu_util import config_canvas, render

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _views(n):
    rng = np.random.default_rng(n)
    cams, off = [], 0
    for i in range(n):
        w, h = int(rng.integers(1, 40)), int(rng.integers(1, 40))
        eye = np.zeros(3) if i % 5 == 1 else rng.uniform(-0.9, 0.9, 3)      # on the mid-planes, inside, outside
        cams.append(synth.look_at_camera(eye, [0.3, 0.1, 0.4], [0, 1, 0], 1.0, w, h, off, (0.1, 0.2, 0.3, 1.0)))
        off += w * h
    return synth.cameras_array(cams)


@pytest.mark.parametrize("n", [1, 4, 5, 64, 65])
def test_arguments_and_staging_agree(n):
    cv, cams = config_canvas(0), _views(n)
    staged, _ = render(cv, cams, key="c0", use_graph=1)
    for kw in (dict(), dict(per_view=1)):
        for _ in range(2):                       # (the second finds the first one's counters in the scratch)
            img, stats = render(cv, cams, key="c0", **kw)
            assert np.array_equal(img, staged), kw
    if n > 64:
        return
    nodes = torch.from_numpy(np.ascontiguousarray(cv.nodes)).cuda()
    leaves = torch.from_numpy(np.ascontiguousarray(cv.leaves).view(np.int16)).cuda()
    args = (nodes, cv.n_records, leaves, cv.n_leaves, cv.depth, cv.extent, cams)
    direct = torch.zeros((len(staged), 4), device="cuda")
    cx.render_noalloc(*args, direct)
    captured = torch.zeros_like(direct)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        cx.render_noalloc(*args, captured)
    for _ in range(2):
        captured.zero_()
        graph.replay()
        assert torch.equal(captured, direct)
