"""Where class products are used: by the class nodes that their tiles take off
the FP64 kernels, seen in the launches of a sweep (3D: residual, patch apply,
and a second launch where the apply is divided).  Many small obstacles leave
few class nodes in many tiles; there the FP64 kernel alone is faster."""
import dataclasses

import numpy as np
import pytest

from paper_2403_11636_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fc():
    from paper_2403_11636_gb300 import fc as m
    return m


def class_products(fc, p, monkeypatch, call):
    """Whether `call` uses class products: one whose wait is 0 reports it."""
    monkeypatch.setenv("FC_DIGIT_WAIT_NS", "0")
    s = fc.Solver(p)
    monkeypatch.delenv("FC_DIGIT_WAIT_NS")
    call(s, s.zeros() + 1.5)
    try:
        s.sync()
    except fc.FcError as e:
        assert e.code == fc.FC_ERR_TIMEOUT
        return True
    finally:
        s.close()
    return False


def sweep_launches(fc, p):
    s = fc.Solver(p)
    x, b = s.zeros(), s.rhs()
    before = fc.launch_count()
    s.smooth_(x, b)
    n = fc.launch_count() - before
    s.close()
    return n


@pytest.mark.parametrize("n, nlevels, spheres, launches", [
    (48, 5, 0, 3), (48, 5, 12, 3), (48, 5, 40, 2), (48, 5, 100, 2), (56, 4, 40, 3), (56, 4, 100, 2),
    (64, 5, 40, 3), (64, 5, 100, 2), (40, 4, 0, 2)])
def test_line_3d(fc, n, nlevels, spheres, launches):
    p = inputs.porous_3d(3, n=n, nspheres=max(spheres, 1), nlevels=nlevels)
    if spheres == 0:
        p = dataclasses.replace(p, shapes=np.zeros((0, 9)))
    assert sweep_launches(fc, p) == launches


@pytest.mark.parametrize("n, nlevels, radius, apply, operator", [
    (192, 6, 0.2, False, False), (256, 6, 0.2, True, False), (256, 6, 0.35, False, False), (384, 6, 0.2, True, True), (512, 7, 0.2, True, True),
    (1024, 8, 0.2, True, True), (1024, 8, 0.48, True, True)])
def test_line_2d(fc, n, nlevels, radius, apply, operator, monkeypatch):
    """(A patch apply meets the right-hand side of x = 0, smoothed once.)"""
    p = inputs.channel_2d(0, n=n, nlevels=nlevels, radius=radius)
    assert class_products(fc, p, monkeypatch, lambda s, x: s.smooth(s.zeros(), x)) == apply
    assert class_products(fc, p, monkeypatch, lambda s, x: s.apply(x)) == operator
