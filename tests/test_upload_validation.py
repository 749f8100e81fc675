"""canvox_upload_octree's validation (Sec. 4.1.1: index pools, eight children per allocation unit) runs on the host's
cores in pieces of the pools; the error it reports must be the one of a sequential walk in pool order. Needs no GPU:
an invalid pool is refused before the device is touched."""
import random

import numpy as np
import pytest

import paper_1704_02724_gb300 as cx
import synth
from paper_1704_02724_gb300 import canvox


def _sequential(nodes, leaves, depth):
    """Message of the first fault in pool order, None for a valid pool."""
    n_rec, n_leaf = len(nodes), len(leaves)
    level, next_rec, next_leaf = [0] * n_rec, 1, 0
    for r in range(n_rec):
        if r >= next_rec:
            return f"record {r} is not referenced before it appears"
        for k in range(8):
            v = int(nodes[r, k])
            if v > 0:
                if v != next_rec:
                    return f"record {r} slot {k}: child {v}, expected {next_rec} (breadth-first order)"
                if v >= n_rec:
                    return f"record {r} slot {k}: child {v} out of range"
                if level[r] + 1 > depth - 1:
                    return f"record {v} at level {level[r] + 1} exceeds depth {depth}"
                level[v] = level[r] + 1
                next_rec += 1
            elif v < 0:
                if -v - 1 != next_leaf:
                    return f"record {r} slot {k}: leaf {-v - 1}, expected {next_leaf} (breadth-first order, modulo 2^31)"
                if next_leaf >= n_leaf:
                    return f"record {r} slot {k}: leaf {next_leaf} out of range"
                next_leaf += 1
    if next_rec != n_rec:
        return f"{n_rec - next_rec} records unreachable"
    if next_leaf != n_leaf:
        return f"{n_leaf - next_leaf} leaves unreferenced"
    q = leaves.astype(np.int64)
    for i in np.flatnonzero(np.any((q >> 10 & 31) == 31, axis=1) | ((q[:, 3] & 0x8000 != 0) & (q[:, 3] & 0x7FFF != 0))):
        return f"leaf {i}: " + ("non-finite FP16" if np.any((q[i] >> 10 & 31) == 31) else "negative extinction")
    return None


@pytest.fixture(scope="module")
def canvas():
    from paper_1704_02724_gb300 import _build
    _build.build()
    rng = np.random.default_rng(2)
    n = 60
    return synth.stamp_canvas(8, 1.0, rng.uniform(-0.5, 0.5, (n, 3)), rng.uniform(0.01, 0.06, n),
                              np.c_[rng.uniform(0, 1, (n, 3)), rng.uniform(0, 9, n)].astype(np.float32))


@pytest.mark.parametrize("seed", range(24))
def test_first_fault_in_pool_order(canvas, seed):
    assert canvas.n_records > 2 * 8192        # several pieces
    r = random.Random(seed)
    nodes, leaves, depth = canvas.nodes.copy(), canvas.leaves.copy(), canvas.depth
    for _ in range(r.choice((1, 1, 3))):
        kind = r.randrange(6)
        i, k = r.randrange(len(nodes)), r.randrange(8)
        if kind == 0:
            nodes[i, k] = 0
        elif kind == 1:
            nodes[i, k] += r.choice((-1, 1))
        elif kind == 2:
            nodes[i, k] = r.choice((len(nodes), 5, -7))
        elif kind == 3:
            depth = r.randint(5, 8)
        elif kind == 4:
            leaves[r.randrange(len(leaves)), r.randrange(4)] = r.choice((0x7C00, 0x7E01, 0xFC00))
        else:
            leaves[r.randrange(len(leaves)), 3] = r.choice((0x8001, 0x8000))
    want = _sequential(nodes, leaves, depth)
    if want is None:
        return   # (for a valid pool the outcome is the device's)
    with pytest.raises(cx.CanvoxError) as e:
        cx.upload_octree(nodes, leaves, depth, 1.0)
    assert e.value.code == canvox.ERR_BAD_TREE and str(e.value).endswith(want)


@pytest.mark.parametrize("cut", ["records", "leaves", "more_leaves"])
def test_pool_sizes(canvas, cut):
    nodes, leaves = canvas.nodes, canvas.leaves
    if cut == "records":
        nodes = nodes[:-1]
    elif cut == "leaves":
        leaves = leaves[:-1]
    else:
        leaves = np.concatenate([leaves, leaves[:2]])
    with pytest.raises(cx.CanvoxError) as e:
        cx.upload_octree(nodes, leaves, canvas.depth, 1.0)
    assert e.value.code == canvox.ERR_BAD_TREE and str(e.value).endswith(_sequential(nodes, leaves, canvas.depth))
