"""Axis-parallel rays beside cell planes (Sec. 6.2: a ray that a plane never meets stays on its side). A ray with a zero
direction component runs in one column of cells to its end; the mixed traversal's FP32 exit times must leave that axis
to "never" wherever the eye is within its unit of 2^-31 of the canvas side, the half unit below a plane among it."""
import math
import random
from fractions import Fraction as Q

import numpy as np
import pytest

import oracle
import paper_1704_02724_gb300 as cx
import synth
from gpu_util import TOL, max_err, render
from synth import random_tree as rt
from test_screens import fma, r32

BIG = r32(Q(10) ** 28)   # the kernel's time per unit of an axis that is never crossed
BG = (0.1, 0.2, 0.3, 1.0)


def test_anchor_of_a_zero_axis():
    """D = X + s - A is at least 1 for the unit the eye is in, so the far face's time D * BIG passes every time that
    another axis can have; the nearest unit gives time 0 for eyes in the half unit below a plane."""
    rng = random.Random(5)
    nearest_fails = 0
    for _ in range(4000):
        sh = rng.randint(1, 30)
        s = 1 << sh
        X = rng.randrange(0, 1 << (31 - sh)) * s
        far = X + s
        gap = Q(rng.choice((0.5, 0.49, 0.01, 2.0 ** -40, 1e-300))) if rng.random() < 0.5 else Q(rng.uniform(0, 1)) * s
        pos = far - gap if rng.random() < 0.8 else Q(X)      # in [X, X + s): a plane belongs to its high side
        k = (pos + Q(1, 2)).__floor__()
        A = min(max(k, 1), 2 ** 31 - 1)
        A -= pos - A < 0
        assert A <= pos and far - A >= 1
        assert fma(r32(Q(far - A)), BIG, Q(0)) >= BIG > 2 ** 31 * Q(2, 2 ** 31)   # times of |d_a| >= 1/2 stay below 2
        # the descent's interval around the anchor holds the unit the ray is in
        assert A - 1 <= pos.__floor__() <= A or A == 1
        nearest_fails += far - k == 0
    assert nearest_fails > 100


def _embedded(level):
    """A depth-4 random scene as one cell at `level` of a 40 km canvas."""
    extent, cell = 40000.0, (2 ** (level - 1) + 12345, 2 ** (level - 1) - 777, 2 ** (level - 2) + 5)
    side = extent * 2.0 ** -level

    def scale(t):
        if isinstance(t, list):
            return [scale(c) for c in t]
        return None if t is None else (t[0], t[1], t[2], t[3] / side)
    small = scale(rt.random_nested(4, seed=91, p_refine=0.6, sigma_range=(0.5, 20.0)))
    cv = rt.from_nested(rt.embed(small, 4, level, cell), level + 4, extent)
    return cv, np.array([-0.5 * extent + c * side for c in cell]), side


def _views(rng, n, lo, side, extent, depth):
    """Axis-parallel views of 3 x 3, 1 x 3 and 3 x 1 pixels (two and one zero components in the middle) from eyes 0.01 to
    0.5 units below and above cell planes of the scene, on them, and anywhere, inside and outside the canvas."""
    unit, cell = extent * 2.0 ** -31, extent * 2.0 ** -depth
    cams, off = [], 0
    for i in range(n):
        ax = i % 3
        eye = lo + rng.integers(0, round(side / cell), 3) * cell
        eye = eye + rng.choice([-0.5, -0.49, -0.3, -0.01, 0.0, 0.01, 0.3, 0.49], 3) * unit
        if i % 5 == 0:
            eye = lo + rng.random(3) * side
        f, up = np.zeros(3), np.zeros(3)
        f[ax] = rng.choice([-1.0, 1.0])
        tan = 0.3
        if i % 4 == 3:
            eye[ax], tan = -f[ax] * extent * (0.5 + rng.random()), 0.3 * side / extent
        up[(ax + 1) % 3] = 1.0
        w, h = ((3, 3), (1, 3), (3, 1))[i // 3 % 3]
        cams.append(synth.camera(eye, np.cross(f, up), up, f, tan, w, h, off, BG))
        off += w * h
    return synth.cameras_array(cams)


@pytest.mark.gpu
@pytest.mark.parametrize("level", [20, 23, 26])
def test_axis_parallel_views_beside_planes(level):
    cv, lo, side = _embedded(level)
    cams = _views(np.random.default_rng(level), 240, lo, side, cv.extent, cv.depth)
    ref = oracle.render(cv, cams)
    for kw in (dict(), dict(traversal=1), dict(frame_levels=3), dict(per_view=1), dict(precision=cx.PREC_FP64_LINKS)):
        img, _ = render(cv, cams, key=("zero axis", level), **kw)
        assert max_err(img, ref) <= TOL, kw


@pytest.mark.gpu
@pytest.mark.parametrize("extent", [1.0, 40000.0])
def test_eye_beside_a_mid_plane(extent):
    """Eyes at rounding noise to half a unit beside the canvas's centre planes, other mid-planes and its faces."""
    import torch
    cv = rt.random_tree(7, seed=91, p_refine=0.6, extent=extent)
    cams, off = [], 0
    for z in (0.0, 0.25, -0.125, -0.5, 0.5):   # (the last two: the canvas's faces)
        for d in (-0.5, -0.3, -1e-6, -1e-8, 0.0, 1e-8, 0.3, 0.5):
            x = (z + d * 2.0 ** -31) * extent
            for eye, f in (([-0.9, 0.03, x / extent], (1.0, 0.0, 0.0)), ([0.03, x / extent, 0.04], (0.0, 0.0, -1.0)),
                           ([x / extent, x / extent, 0.04], (0.0, 0.0, 1.0))):
                cams.append(synth.camera(np.array(eye) * extent, np.cross(f, (0, 1, 0)), (0, 1, 0), f, 0.4, 5, 5, off, BG))
                off += 25
    cams = synth.cameras_array(cams)
    ref = oracle.render(cv, cams)
    for kw in (dict(), dict(traversal=1), dict(precision=cx.PREC_FP64_LINKS)):
        img, _ = render(cv, cams, key=("mid-plane", extent), **kw)
        assert max_err(img, ref) <= TOL, kw
    nodes = torch.from_numpy(np.ascontiguousarray(cv.nodes)).cuda()
    leaves = torch.from_numpy(np.ascontiguousarray(cv.leaves).view(np.int16)).cuda()
    out = torch.empty((32, 4), device="cuda")
    part = cams[6:7].copy()
    part["out_offset_px"] = 0
    cx.render_noalloc(nodes, cv.n_records, leaves, cv.n_leaves, cv.depth, cv.extent, part, out)
    torch.cuda.synchronize()
    assert max_err(out[:25].cpu().numpy().astype(np.float64), ref[150:175]) <= TOL
