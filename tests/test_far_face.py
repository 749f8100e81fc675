"""Leaves at the canvas's far faces, reached from its near ones with the anchor still there (Sec. 6.2: the exit of the
canvas): the way is up to 2^31 - 1 units, whose FP32 value is 2^31, one past the largest integer."""
import random
from fractions import Fraction as Q

import numpy as np
import pytest

import oracle
import paper_1704_02724_gb300 as cx
import synth
from gpu_util import TOL, max_err, render
from synth import random_tree as rt
from test_position_screens import rest_time, split_inv
from test_screens import add, fma, mul, r32, sub

TOP = 2 ** 31 - 1


def _exit_time(D, ih, il, rr, most):
    dh = min(r32(Q(D)), most)
    dl = r32(Q(D - min(int(dh), TOP)))           # (the conversion back saturates)
    p = mul(dh, ih)
    lo = add(fma(dh, il, fma(dl, ih, fma(dh, ih, -p))), rr)
    hi = add(p, lo)
    return hi + sub(lo, sub(hi, p))


def test_exit_time_of_the_longest_ways():
    rng = random.Random(3)
    short = 0
    for _ in range(2000):
        D = TOP - rng.randrange(0, rng.choice((2, 64, 200, 2 ** 20)))
        ih, il = split_inv(rng.uniform(0.5, 1.0))
        rest = Q(rng.uniform(-1.0, 0.5))
        rr, t = rest_time(rest, ih, il), (D - rest) * (ih + il)
        bound = Q(1, 2 ** 44) * t + Q(1, 2 ** 24) * ih
        assert abs(_exit_time(D, ih, il, rr, Q(2 ** 31 - 128)) - t) <= bound
        short += abs(_exit_time(D, ih, il, rr, Q(2 ** 31)) - t) > bound
    assert short > 200                           # without the clamp: a unit short


@pytest.mark.gpu
@pytest.mark.parametrize("level", [14, 18, 21])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_leaf_at_the_far_face(level, axis):
    """Eight leaves of one optical depth per side, in the last cells before the far (and the near) face of one axis, seen
    by single rays that enter through the opposite face."""
    extent = 40000.0
    side = extent * 2.0 ** -level
    for sign in (1.0, -1.0):
        c = [2 ** (level - 1) + 2 ** (level - 2) + 77, 2 ** (level - 1) + 2 ** (level - 3) + 5, 2 ** (level - 1) - 9]
        c[axis] = 2 ** level - 1 if sign > 0 else 0
        cell = tuple(x >> 1 for x in c)
        leaf = (0.9, 0.8, 0.7, 1.0 / side)
        cv = rt.from_nested(rt.embed([leaf] * 8, 1, level - 1, cell), level, extent)
        lo = np.array([-0.5 * extent + 2 * side * x for x in cell])
        rng = np.random.default_rng(level)
        cams = []
        for i in range(100):
            target = lo + rng.uniform(0.1, 1.9, 3) * side
            eye = target + rng.uniform(-0.05, 0.05, 3) * extent
            eye[axis] = -sign * extent * rng.uniform(0.5, 0.9)
            cams.append(synth.look_at_camera(eye, target, np.eye(3)[axis - 1], 1e-9, 1, 1, i, (0.1, 0.2, 0.3, 1.0)))
        cams = synth.cameras_array(cams)
        ref = oracle.render(cv, cams)
        assert np.mean(ref[:, 3] > 0.0) > 0.9    # the rays meet the leaves
        for kw in (dict(), dict(traversal=1), dict(precision=cx.PREC_FP64_LINKS)):
            img, _ = render(cv, cams, key=("far face", level, axis, sign), **kw)
            assert max_err(img, ref) <= TOL, kw
