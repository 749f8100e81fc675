"""Eyes within a unit (2^-31 of the side) of the canvas's faces and a little outside them, looking almost along the face
(Sec. 6.1: the eye keeps its FP64 position): the ray leaves or enters through that face, or meets the first planes, after a
way that depends on the eye's distance from the face, which has to keep a precision of its own."""
import numpy as np
import pytest

import oracle
import paper_1704_02724_gb300 as cx
import synth
from gpu_util import max_err, render
from synth import random_tree as rt

pytestmark = pytest.mark.gpu


def _views(rng, n, extent):
    half, unit = 0.5 * extent, extent * 2.0 ** -31
    cams = []
    for i in range(n):
        a, face = i % 3, (-1.0, 1.0)[i % 2]
        inside = i % 4 < 2
        # the distance from the face is exact: the face and the eye are binary64 numbers
        eye = rng.uniform(-0.45, 0.45, 3) * extent
        eye[a] = face * (half - rng.uniform(0.0, 0.6) * unit * (1.0 if inside else -1.0))
        gap = abs(half - abs(eye[a]))
        f = rng.normal(size=3)
        f[a] = 0.0
        f = f / np.linalg.norm(f)
        # through the face (or back to it from outside) after a fifth to four fifths of a side; some the other way
        f[a] = gap / (rng.uniform(0.2, 0.8) * extent) * face * (1.0 if inside else -1.0) * (1.0 if i % 5 else -1.0)
        up = np.eye(3)[(a + 1) % 3] if abs(f[(a + 1) % 3]) < 0.7 else np.eye(3)[(a + 2) % 3]
        right = np.cross(f, up)
        cams.append(synth.camera(eye, right, np.cross(right, f), f, 1e-3, 1, 1, i, (0.1, 0.2, 0.3, 1.0)))
    return synth.cameras_array(cams)


@pytest.mark.parametrize("extent", [1.0, 5.0, 40000.0])
def test_eyes_beside_faces(extent):
    cv = rt.random_tree(5, seed=7, p_refine=0.5, p_empty=0.1, extent=extent, sigma_range=(0.5 / extent, 5.0 / extent))
    cams = _views(np.random.default_rng(3), 600, extent)
    ref = oracle.render(cv, cams)
    for kw, tol in ((dict(precision=cx.PREC_FP64_LINKS), 1e-6), (dict(), 1e-5), (dict(traversal=1), 1e-5)):
        img, _ = render(cv, cams, key=("face", extent), **kw)
        assert max_err(img, ref) <= tol, kw
