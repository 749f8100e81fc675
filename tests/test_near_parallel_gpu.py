"""Rays almost parallel to an axis's planes (Sec. 6.2: the direction's sign decides on a plane): a component down to
1e-50 of the direction, whose reciprocal leaves the FP32 range, from eyes a fraction of the finest unit beside a
mid-plane, on it, and away from it."""
import numpy as np
import pytest

import oracle
import paper_1704_02724_gb300 as cx
import synth
from gpu_util import TOL, max_err, render
from synth import random_tree as rt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dz", [1e-50, -1e-50, 1e-44, -1e-38, 1e-30, -1e-20])
@pytest.mark.parametrize("extent", [1.0, 40000.0])
def test_component_below_fp32(dz, extent):
    cv = rt.random_tree(7, seed=91, p_refine=0.6, extent=extent)
    cams, off = [], 0
    for z in (0.25, -0.125):                                   # mid-planes; in units of 2^-31 of the side beside them:
        for d in (-3.0, -0.3, -1e-6, 0.0, 1e-6, 0.3, 2.0):
            cam = synth.look_at_camera([-0.9 * extent, 0.03 * extent, (z + d * 2.0 ** -31) * extent], [extent, 0.0, 0.0],
                                       [0, 1, 0], 0.4, 1, 24, off, (0.1, 0.2, 0.3, 1.0))
            cam["forward"], cam["up"], cam["right"] = (1.0, 0.0, dz), (0.0, 1.0, 0.0), (0.0, 0.0, 1.0)
            cams.append(cam)                                   # one column: x = 0, so d_z is the forward's
            off += 24
    cams = synth.cameras_array(cams)
    ref = oracle.render(cv, cams)
    for kw in (dict(), dict(traversal=1), dict(precision=cx.PREC_FP64_LINKS)):
        img, _ = render(cv, cams, key=("near", extent, dz), **kw)
        assert max_err(img, ref) <= TOL, kw
