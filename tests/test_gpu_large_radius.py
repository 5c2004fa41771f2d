"""Obstacles so large that their boundary rule has more than 2^31 points (a
circle used as a nearly flat wall): the operator against that of a radius just
below.  The two walls differ by a sagitta of at most 4e-7 (2D) and 1e-8 (3D)
over the box, 1e-5 of a cell, so the operators agree to 1e-3 by a wide margin;
with the points cut to 32 bits the wall's terms were missing: 0.03 (2D), 0.002
(3D)."""
import dataclasses

import numpy as np
import pytest

from paper_2403_11636_gb300 import inputs
from tests.gpu_util import rel

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fc():
    from paper_2403_11636_gb300 import fc as m
    return m


def wall(kind, f):
    """A wall at 0.4 whose rule has f 2^31 points at quadrature depth 6."""
    if kind == "sphere":
        r = f * 2.0 ** 31 / (2 * 64 * 2 * np.pi * 8)
        shape = [0.0, 0.4 - r, 0.52, 0.47, r, r, r, 1.0, 0.0]
        return dataclasses.replace(inputs.channel_3d(0, n=8, nlevels=2, qdepth=6), shapes=np.array([shape]))
    r = f * 2.0 ** 31 / (8 * 64 * 2 * np.pi * 32)
    if kind == "circle":
        shape = [0.0, 0.52, 0.4 - r, 0.0, r, r, r, 1.0, 0.0]
    else:
        shape = [1.0, 0.4 - r, 0.47, 0.0, r, 0.75 * r, 0.0, 1.0, 0.0]
    return dataclasses.replace(inputs.channel_2d(0, n=32, nlevels=3, qdepth=6), shapes=np.array([shape]))


@pytest.mark.parametrize("kind", ["circle", "ellipse", "sphere"])
def test_more_points_than_32_bits(fc, kind):
    p, q = wall(kind, 0.98), wall(kind, 1.02)
    x = inputs.random_vector(p, 4)
    free = np.repeat(np.array([1.0, 0.0]), [p.dim, 1])  # velocities alone: the Nitsche terms stand out
    x = x * np.tile(free, len(x) // (p.dim + 1))
    below, above = (fc.Solver(k).apply(x).cpu().numpy() for k in (p, q))
    assert rel(above, below) <= 1e-3
