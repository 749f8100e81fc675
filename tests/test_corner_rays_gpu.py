"""Rays from far eyes through exact corners and edges of cells (Sec. 6.2: two or three faces are met at one time): the FP64 times
of a far eye's ray differ there by more than a position next to its anchor is resolved, so a plane can come out a little
before the one just crossed, and the ray must stay in its column of cells all the same."""
import numpy as np
import pytest

import oracle
import paper_1704_02724_gb300 as cx
import synth
from gpu_util import TOL, max_err, render
from synth import random_tree as rt

pytestmark = pytest.mark.gpu


def _views(rng, n, depth, extent, far):
    cams = []
    for i in range(n):
        lev = rng.integers(1, depth + 1)
        corner = (rng.integers(0, 2 ** lev + 1, 3) / 2.0 ** lev - 0.5) * extent
        f = np.sign(rng.normal(size=3)) if i % 3 else rng.normal(size=3)
        f = f / np.linalg.norm(f)
        if i % 4 == 0:                                     # through an edge
            corner[rng.integers(0, 3)] += rng.uniform(-0.1, 0.1) * extent
        up = np.eye(3)[np.argmin(np.abs(f))]
        cams.append(synth.look_at_camera(corner - f * far * extent, corner, up, 0.4, 1, 1, i, (0.1, 0.2, 0.3, 1.0)))
        cams[-1]["forward"] = f                            # (as drawn: the eye is on the corner's line)
    return synth.cameras_array(cams)


@pytest.mark.parametrize("extent", [1.0, 1000.0])
@pytest.mark.parametrize("far", [2.0, 100.0])
def test_corners(extent, far):
    cv = rt.random_tree(6, seed=31, p_refine=0.55, extent=extent, sigma_range=(0.2 / extent, 20.0 / extent))
    cams = _views(np.random.default_rng(int(far)), 3000, 6, extent, far)
    ref = oracle.render(cv, cams)
    for kw in (dict(frame_levels=1), dict(frame_levels=2, traversal=1), dict(), dict(traversal=1),
               dict(precision=cx.PREC_FP64_LINKS)):
        img, _ = render(cv, cams, key=("corners", extent, far), **kw)
        assert max_err(img, ref) <= TOL, kw
