"""canvox_upload_octree refuses a canvas deeper than it says at the first record past that level (Sec. 4.1.1: a bounded
depth), however long the chain of records is. Needs no GPU: an invalid pool is refused before the device is touched."""
import time

import numpy as np
import pytest

import paper_1704_02724_gb300 as cx
from paper_1704_02724_gb300 import canvox


@pytest.fixture(scope="module", autouse=True)
def _built():
    from paper_1704_02724_gb300 import _build
    _build.build()


def _chain(n, slot=0):
    nodes = np.zeros((n, 8), dtype=np.int32)
    nodes[:-1, slot] = np.arange(1, n)
    return nodes


@pytest.mark.parametrize("depth,n,slot", [(1, 2, 0), (1, 20000, 7), (8, 9, 3), (8, 20000, 0), (30, 31, 5), (30, 100000, 0)])
def test_chain_message(depth, n, slot):
    """A chain of n records is n levels: record `depth` is the first too deep."""
    with pytest.raises(cx.CanvoxError) as e:
        cx.upload_octree(_chain(n, slot), np.zeros((0, 4), dtype=np.uint16), depth, 1.0)
    assert e.value.code == canvox.ERR_BAD_TREE
    assert str(e.value).endswith(f"record {depth} at level {depth} exceeds depth {depth}")


def test_long_chain_is_refused_at_once():
    """Two million records (64 MB): a walk of the pool takes milliseconds, a piece of it for every level 12 s of one core."""
    nodes, leaves = _chain(2_000_000), np.zeros((0, 4), dtype=np.uint16)
    t = time.thread_time()          # the calling thread's
    with pytest.raises(cx.CanvoxError):
        cx.upload_octree(nodes, leaves, 30, 1.0)
    assert time.thread_time() - t < 2.0
