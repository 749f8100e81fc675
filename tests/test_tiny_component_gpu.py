"""Direction components whose reciprocal leaves the binary64 range (Sec. 6.2: the direction's sign decides on a plane):
such an axis is never crossed, and its infinite time must not be taken for the first one."""
import numpy as np
import pytest

import oracle
import paper_1704_02724_gb300 as cx
import synth
from gpu_util import TOL, max_err, render
from synth import random_tree as rt

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dz", [1e-310, -1e-310, 5e-324, -5e-324, 1e-300, -1e-300, 1e-290])
@pytest.mark.parametrize("extent", [1.0, 40000.0])
def test_component_without_reciprocal(dz, extent):
    cv = rt.random_tree(7, seed=91, p_refine=0.6, extent=extent)
    cams = []
    for z in (0.25, -0.125, -0.4371):
        for d in (-3.0, -0.3, 0.0, 0.3, 2.0):      # units of 2^-31 of the side beside a mid-plane
            for eye in ([-0.9, 0.03], [0.07, -0.21]):
                at = np.array([eye[0], eye[1], z + d * 2.0 ** -31]) * extent
                for row in range(3):
                    y = (0.0, 0.13, -0.2)[row]
                    n = np.hypot(1.0, y)
                    cams.append(synth.camera(at, (0.0, 0.0, 1.0), (-y / n, 1.0 / n, 0.0), (1.0 / n, y / n, dz), 0.1, 1, 1,
                                             len(cams), (0.1, 0.2, 0.3, 1.0)))
    cams = synth.cameras_array(cams)               # single pixels: d_z is the forward's
    ref = oracle.render(cv, cams)
    for kw in (dict(precision=cx.PREC_FP64_LINKS), dict(), dict(traversal=1)):
        img, _ = render(cv, cams, key=("tiny", extent, dz), **kw)
        assert max_err(img, ref) <= TOL, kw
