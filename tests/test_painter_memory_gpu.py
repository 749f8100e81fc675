"""The device memory that the painter keeps for the next paint follows the last two paintings: small ones after a large one
give the large one's back, without a call to the allocator failing first."""
import numpy as np
import pytest

import paper_1704_02724_gb300 as cx
from gpu_util import _uploaded

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
MIB = 1 << 20


def _stamps(n, seed):
    rng = np.random.default_rng(seed)
    return (rng.uniform(-0.45, 0.45, (n, 3)), rng.uniform(0.004, 0.012, n),
            np.c_[rng.uniform(0, 1, (n, 3)), rng.uniform(0, 9, n)].astype(np.float32))


def _used():
    torch.cuda.synchronize()
    free, total = torch.cuda.mem_get_info()
    return total - free


def test_small_paintings_after_a_large_one():
    _uploaded["key"] = None
    cx.release()
    small, large = _stamps(20, 1), _stamps(30000, 2)
    cx.paint_spheres(10, 1.0, *small)
    base = _used()
    cx.paint_spheres(10, 1.0, *large)
    held = _used() - base
    assert held > 1024 * MIB              # (the large painting's own canvas and what is kept of its levels)
    cx.paint_spheres(10, 1.0, *large)     # the same again
    assert abs(_used() - base - held) <= held // 4
    cx.paint_append(*_stamps(5, 3))       # (an append belongs to its painting)
    assert _used() - base >= held // 2
    for _ in range(2):
        cx.paint_spheres(10, 1.0, *small)
    assert _used() - base <= 128 * MIB    # 64 MiB for gaps, in blocks of 32 MiB
    cx.release()
