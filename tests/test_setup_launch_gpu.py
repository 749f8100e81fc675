"""A render's set-up (Sec. 4.1.5: views and starting cells before the rays): up to 64 views travel as the arguments of
one launch, in two sizes of argument block; more views, and renders replayed from a graph, are staged in pinned memory.
Either way the rays get the same words, so the images are equal bit for bit."""
import numpy as np
import pytest

import oracle
import paper_1704_02724_gb300 as cx
import synth
from gpu_util import TOL, config_canvas, max_err, render
from synth import random_tree as rt

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


@pytest.mark.parametrize("extent,depth", [(1.0, 8), (40000.0, 30), (1000.0, 3)])
def test_eyes_beside_planes(extent, depth):
    """The eye's leaf from its position in units of 2^-31 of the side: eyes on mid-planes of every level, a fraction of a
    unit or an ulp beside them, and within a unit of the canvas's faces."""
    cv = rt.random_tree(min(depth, 9), seed=17, p_refine=0.6, extent=extent)
    rng = np.random.default_rng(depth)
    unit, cams, off = extent * 2.0 ** -31, [], 0
    for i in range(60):
        lev = rng.integers(1, 12, 3)
        plane = (rng.integers(0, 2 ** lev) / 2.0 ** lev - 0.5) * extent
        beside = rng.choice([0.0, 0.25, -0.25, 0.5, -0.5, 1e-7, -1e-7, 3.0, -1.0], 3) * unit
        eye = np.where(rng.random(3) < 0.7, plane + beside, rng.uniform(-0.5, 0.5, 3) * extent)
        eye = np.nextafter(eye, rng.choice([-1.0, 1.0], 3) * extent) if i % 3 == 0 else eye
        if i % 10 == 0:
            eye[i // 10 % 3] = rng.choice([-0.5, 0.5]) * (extent - 2 * abs(beside[0]))
        cams.append(synth.look_at_camera(eye, rng.uniform(-0.4, 0.4, 3) * extent, [0, 1, 0], 1.0, 8, 4, off,
                                         (0.1, 0.2, 0.3, 1.0)))
        off += 32
    cams = synth.cameras_array(cams)
    ref = oracle.render(cv, cams)
    for kw in (dict(), dict(use_graph=1), dict(precision=cx.PREC_FP64_LINKS)):
        img, _ = render(cv, cams, key=("planes", extent, depth), **kw)
        assert max_err(img, ref) <= TOL, kw
