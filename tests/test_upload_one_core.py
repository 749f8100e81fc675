"""A process held to one core validates and hashes an upload on one walk by itself (Sec. 4.1.1: index pools); messages,
hash and links are those of the host's team of threads."""
import contextlib
import os
import random

import numpy as np
import pytest

import paper_1704_02724_gb300 as cx
import synth
from paper_1704_02724_gb300 import canvox
from test_upload_validation import _sequential


@contextlib.contextmanager
def one_core():
    before = os.sched_getaffinity(0)
    os.sched_setaffinity(0, {min(before)})
    try:
        yield
    finally:
        os.sched_setaffinity(0, before)


@pytest.fixture(scope="module")
def pools():
    from paper_1704_02724_gb300 import _build
    _build.build()
    rng = np.random.default_rng(2)
    n = 60
    return synth.stamp_canvas(8, 1.0, rng.uniform(-0.5, 0.5, (n, 3)), rng.uniform(0.01, 0.06, n),
                              np.c_[rng.uniform(0, 1, (n, 3)), rng.uniform(0, 9, n)].astype(np.float32))


def _message(nodes, leaves, depth):
    with pytest.raises(cx.CanvoxError) as e:
        cx.upload_octree(nodes, leaves, depth, 1.0)
    assert e.value.code == canvox.ERR_BAD_TREE
    return str(e.value)


@pytest.mark.parametrize("seed", range(16))
def test_messages(pools, seed):
    r = random.Random(100 + seed)
    nodes, leaves, depth = pools.nodes.copy(), pools.leaves.copy(), pools.depth
    i, k, kind = r.randrange(len(nodes)), r.randrange(8), seed % 4
    if kind == 0:
        nodes[i, k] += r.choice((-1, 1))
    elif kind == 1:
        depth = r.randint(4, 7)
    elif kind == 2:
        for _ in range(3):                                  # the first in pool order is reported
            leaves[r.randrange(len(leaves)), 3] = r.choice((0x8001, 0x7C00))
    else:
        nodes, leaves = (nodes[:-1], leaves) if seed % 8 == 3 else (nodes, leaves[:-1])
    want = _sequential(nodes, leaves, depth)
    if want is None:
        return   # (-0 or an empty slot: a valid pool)
    with one_core():
        alone = _message(nodes, leaves, depth)
    assert alone.endswith(want) and alone == _message(nodes, leaves, depth)


@pytest.mark.gpu
@pytest.mark.parametrize("levels", [1, 2, 8])
def test_hash_and_image(pools, levels):
    import gpu_util
    import torch
    from synth import random_tree as rt
    gpu_util._uploaded["key"] = None                        # (the canvas is replaced here)
    cv = pools if levels == 8 else rt.random_tree(levels, seed=5, p_refine=0.9)
    cams = synth.cameras_array([synth.look_at_camera([1.1, 0.7, -1.3], [0, 0, 0], [0, 1, 0], 0.5, 64, 48)])
    got = []
    for scope in (one_core, contextlib.nullcontext):
        with scope():
            cx.upload_octree(cv.nodes, cv.leaves, cv.depth, cv.extent)
        hashes, out = cx.octree_hash(), torch.empty((64 * 48, 4), device="cuda")
        cx.render(cams, out)                                # (by the neighbour links, level by level)
        torch.cuda.synchronize()
        assert hashes[0] == hashes[1] != 0
        got.append((hashes, out))
    assert got[0][0] == got[1][0] and torch.equal(got[0][1], got[1][1])
