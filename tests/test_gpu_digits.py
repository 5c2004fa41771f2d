"""Class products on the tensor cores (fc_digits.cu) against the oracle and the
general kernels.

Large levels take the products of uncut, unconstrained nodes from exact digit
products; the others stay in FP64.  Sizes at the edges of the tiles (32 x 14
and 16 x 8 x 4 nodes), both classes, ragged and anisotropic grids, and
values at which a tile's common exponent could go wrong: a wide range of
magnitudes inside a tile, zeros, and an infinity.  Bounds as in the parity
tests: operator 1e-12, sweep 1e-10 relative."""
import dataclasses

import numpy as np
import pytest

from oracle import oracle as O
from paper_2403_11636_gb300 import inputs
from tests.gpu_util import rel

pytestmark = pytest.mark.gpu

SWEEP_TOL = 1e-10
OPER_TOL = 1e-12

CIRCLE = np.array([[0.0, 0.55, 0.45, 0.0, 0.3, 0.3, 0.3, 1.0, 0.0]])  # room for fictitious class patches
BALL = np.array([[0.0, 0.5, 0.45, 0.5, 0.42, 0.42, 0.42, 1.0, 0.0]])


def square(nx, ny, nlevels=2, **kw):
    return dataclasses.replace(inputs.channel_2d(0, n=64, nlevels=nlevels), **{"n": (nx, ny), "shapes": CIRCLE, **kw})


def cube(n, nlevels=2, **kw):
    return dataclasses.replace(inputs.porous_3d(0, n=8, nspheres=1, nlevels=nlevels), n=n, shapes=BALL, **kw)


PROBS = {                                         # (apply from 50,000 nodes, residual from 130,000)
    "232x256": square(232, 256, nlevels=4),       # class nodes end one row into a last tile
    "384x352": square(384, 352, nlevels=5),
    "528x272": square(528, 272, nlevels=5, hi=(2.2, 0.41),
                      shapes=np.array([[1.0, 0.9, 0.2, 0.0, 0.15, 0.08, 0.0, 0.8, 0.6]])),
    "free": square(368, 368, nlevels=5, preset=2),  # no constrained nodes
    "empty": dataclasses.replace(square(256, 256, nlevels=4), shapes=np.zeros((0, 9))),
}
PROBS3 = {                                        # against the FP64 kernels of a batch of one
    "48": cube((48, 48, 48), nlevels=4),          # 45 layers of class patches: a last tile of one
    "48x40x56": cube((48, 40, 56), nlevels=4, hi=(1.2, 1.0, 1.4)),
    "pores": inputs.porous_3d(3, n=48, nspheres=12, nlevels=4),
}


@pytest.fixture(scope="module")
def fc():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2403_11636_gb300 import build, fc as fcmod
    build.build()
    return fcmod


def fields(L, kind, seed):
    n = L.ndof if isinstance(L.ndof, int) else int(L.ndof)
    x = inputs.uniform_array(n, seed)
    if kind == "wide":                            # magnitudes over 12 decades within every tile
        x = x * 10.0 ** (12.0 * inputs.uniform_array(n, seed + 1, -0.5, 0.5))
    elif kind == "zeros":
        x = np.where(inputs.uniform_array(n, seed + 1) > 0.98, x, 0.0)
    return x


@pytest.mark.parametrize("kind", ["plain", "wide", "zeros"])
@pytest.mark.parametrize("name", list(PROBS))
def test_class_products(fc, name, kind):
    p = PROBS[name]
    L = O.Level.from_problem(p)
    A, b, _ = L.csr()
    s = fc.Solver(p)
    assert s.ndof() == L.ndof and s.ndof() // 3 >= 50000
    x = fields(L, kind, 5)
    assert rel(s.apply(x).cpu().numpy(), A @ x) <= OPER_TOL
    want = L.sweep(b, x) - x
    assert rel(s.smooth(x, b).cpu().numpy() - x, want) <= SWEEP_TOL
    assert rel(s.residual(x, b).cpu().numpy(), b - A @ x) <= OPER_TOL


@pytest.mark.parametrize("kind", ["plain", "wide", "zeros"])
@pytest.mark.parametrize("name", list(PROBS3))
def test_class_products_3d(fc, name, kind):
    """3D patch apply: the general FP64 kernels round each of 402 partial sums
    (4.5e-14 of the sum of magnitudes, about 100 times the update where alpha-
    scaled rows cancel), so the two agree to 1e-11."""
    import torch
    p = PROBS3[name]
    s = fc.Solver(p)
    n = s.ndof()
    assert n // 4 >= 100000
    x = inputs.uniform_array(n, 5)
    if kind == "wide":
        x = x * 10.0 ** (12.0 * inputs.uniform_array(n, 6, -0.5, 0.5))
    elif kind == "zeros":
        x = np.where(inputs.uniform_array(n, 6) > 0.98, x, 0.0)
    b = inputs.uniform_array(n, 7)
    got = s.smooth(x, b).cpu().numpy()
    B = fc.Batch([s], tile=(8, 256, 4))
    want = torch.as_tensor(x).cuda()
    B.smooth_(want, torch.as_tensor(b).cuda())
    want = want.cpu().numpy()
    assert rel(got - x, want - x) <= 1e-11
    B.close()


@pytest.mark.parametrize("name", ["384x352"])
def test_class_products_dedup_and_repeat(fc, name):
    """One block per patch gives the same values, and so does a second run."""
    p = PROBS[name]
    s1, s0 = fc.Solver(p, dedup=1), fc.Solver(p, dedup=0)
    x, b = inputs.random_vector(p, 7), inputs.random_vector(p, 8)
    y = s1.smooth(x, b, nsweeps=2).cpu().numpy()
    np.testing.assert_array_equal(y, s1.smooth(x, b, nsweeps=2).cpu().numpy())
    np.testing.assert_array_equal(y, s0.smooth(x, b, nsweeps=2).cpu().numpy())


@pytest.mark.parametrize("name", ["384x352"])
def test_class_products_not_finite(fc, name):
    """An infinity or NaN reaches the nodes whose rows read it, and no other."""
    p = PROBS[name]
    L = O.Level.from_problem(p)
    A, _, _ = L.csr()
    s = fc.Solver(p)
    x = inputs.random_vector(p, 9)
    at = (p.dim + 1) * (int(np.prod([k + 1 for k in p.n])) // 2 + 3)
    for bad in (np.inf, np.nan):
        y = x.copy()
        y[at] = bad
        got = s.apply(y).cpu().numpy()
        reads = np.zeros(len(x), bool)
        reads[A.tocsc().indices[A.tocsc().indptr[at]:A.tocsc().indptr[at + 1]]] = True
        clean = np.isfinite(got)
        assert not clean[at]
        near = np.abs(np.arange(len(x)) - at) >= 0
        # rows without an entry for the value are as without it
        keep = clean & ~reads & near
        assert rel(got[keep], (A @ x)[keep]) <= OPER_TOL
        assert np.count_nonzero(~clean) <= (p.dim + 1) * 3 ** p.dim


def test_class_products_extreme_scale(fc):
    """Values whose exponents leave the fixed-point window take plain FP64."""
    p = PROBS["384x352"]
    L = O.Level.from_problem(p)
    A, b, _ = L.csr()
    s = fc.Solver(p)
    x = inputs.random_vector(p, 3)
    for f in (1e-200, 1e200):
        assert rel(s.apply(x * f).cpu().numpy() / f, A @ x) <= OPER_TOL
