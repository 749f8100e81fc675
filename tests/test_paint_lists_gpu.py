"""The device painter at the edges of its list walks (Sec. 5.1-5.2 on the GPU): lists of about eight entries (one load
of an octet), of about 512 (the longest a cell's octet walks), of about a multiple of 128 (an item of a longer one), and
canvases whose lengths leave the FP32 range of the cover screen. The pools equal the host painter's byte for byte."""
import numpy as np
import pytest

import paper_1704_02724_gb300 as cx
import synth
from gpu_util import _uploaded

pytestmark = pytest.mark.gpu


def _check(D, E, c, r, q):
    ref = synth.stamp_canvas(D, E, c, r, q)
    _uploaded["key"] = None
    assert cx.paint_spheres(D, E, c, r, q) == (ref.n_records, ref.n_leaves)
    nodes, leaves = cx.download_octree()
    np.testing.assert_array_equal(nodes, ref.nodes)
    np.testing.assert_array_equal(leaves, ref.leaves)


@pytest.mark.parametrize("n", [1, 7, 8, 9, 127, 129, 511, 512, 513, 640, 641, 1025])
def test_list_lengths(n):
    """Every stamp reaches every octant, so the root and its children carry lists of n entries."""
    rng = np.random.default_rng(n)
    c = rng.uniform(-0.02, 0.02, (n, 3))
    r = np.exp(rng.uniform(np.log(0.02), np.log(0.4), n))
    r[rng.random(n) < 0.1] = 0.9          # covers whole octants (not the corners): painted entries on the way down
    q = np.c_[rng.uniform(0, 1, (n, 3)), rng.uniform(0, 9, n)].astype(np.float32)
    _check(6, 1.0, c, r, q)


@pytest.mark.parametrize("extent", [2.0 ** -140, 2.0 ** -70, 2.0 ** 60, 2.0 ** 120, 2.0 ** 400])
def test_extents_past_the_screen(extent):
    rng = np.random.default_rng(5)
    n = 60
    c = rng.uniform(-0.5, 0.5, (n, 3)) * extent
    r = np.exp(rng.uniform(np.log(0.01), np.log(0.3), n)) * extent
    q = np.c_[rng.uniform(0, 1, (n, 3)), rng.uniform(0, 9, n)].astype(np.float32)
    _check(7, extent, c, r, q)


@pytest.mark.parametrize("n", [2560, 2561, 10241])
def test_item_lengths(n):
    """Lists at the edges between items of 16, 32 and 64 entries."""
    rng = np.random.default_rng(n)
    c = rng.uniform(-0.02, 0.02, (n, 3))
    r = np.exp(rng.uniform(np.log(0.02), np.log(0.4), n))
    q = np.c_[rng.uniform(0, 1, (n, 3)), rng.uniform(0, 9, n)].astype(np.float32)
    _check(4, 1.0, c, r, q)


@pytest.mark.parametrize("n", [100, 200])
def test_planes_through_a_room(n):
    """Small stamps that touch, or miss by a relative 1e-16 to 1e-3, the planes of cells 2^16 times their size: the screen
    next to a far coarser cell's plane, in an octet's own walk and in items."""
    rng = np.random.default_rng(n)
    E, D = 40000.0, 18
    r = rng.uniform(0.8, 2.0, n)
    c = rng.uniform(-8.0, 8.0, (n, 3)) + [E / 8, -E / 4, 0.0]
    a = rng.integers(0, 3, n)
    gap = 10.0 ** rng.uniform(-16, -3, n) * rng.choice([-1.0, 1.0], n)
    c[np.arange(n), a] = np.array([E / 8, -E / 4, 0.0])[a] + rng.choice([-1.0, 1.0], n) * r * (1 + gap)
    q = np.c_[rng.uniform(0, 1, (n, 3)), rng.uniform(0, 9, n)].astype(np.float32)
    _check(D, E, c, r, q)


@pytest.mark.parametrize("depth", [1, 2, 5, 7])
def test_centres_at_the_radius(depth):
    """Stamps whose surface passes exactly, or an ulp inside or outside, through centres of the deepest leaves."""
    rng = np.random.default_rng(depth)
    n, h = 150, 2.0 ** -depth
    c = (rng.integers(0, 2 ** depth, (n, 3)) + 0.5) * h - 0.5             # leaf centres
    r = rng.integers(1, max(2, 2 ** depth // 8), n) * h
    r[::5] = h * np.sqrt(rng.integers(1, 12, len(r[::5])))
    r = r * (1.0 + rng.integers(-1, 2, n) * 2.0 ** -52)
    q = np.c_[rng.uniform(0, 1, (n, 3)), rng.uniform(0, 9, n)].astype(np.float32)
    _check(depth, 1.0, c, r, q)
