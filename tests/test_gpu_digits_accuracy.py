"""Class products node by node: the error of each against its own sum |w||v|,
with values of very different size in a tile (a ramp, spikes, a random exponent
per value, components of different scale).

A chain of n FP64 fused multiply-adds, m additions over the lanes and the last
rounding is off by at most (n + m + 1) 2^-53 sum |w||v|: 15 + 2 + 1 for a 2D patch
row (59 slots, 4 lanes), 51 + 3 + 1 for a 3D one (402, 8), and 3 neighbours of 4
products for the operator, 2 additions, 1 rounding.  The digits' results are held
to the same bounds.  With them relative to the tile's largest value alone, a ramp's nodes are
off by 2^-2 of sum |w||v| and more.  Reference: extended precision, from the
rows that the solver stores."""
import dataclasses

import numpy as np
import pytest

from paper_2403_11636_gb300 import inputs

pytestmark = pytest.mark.gpu

EMPTY2 = dataclasses.replace(inputs.channel_2d(0, n=64, nlevels=5), n=(384, 368), shapes=np.zeros((0, 9)), omega=1.0)
LARGE2 = dataclasses.replace(EMPTY2, n=(768, 672), nlevels=6)   # operator
EMPTY3 = dataclasses.replace(inputs.porous_3d(0, n=8, nspheres=1, nlevels=4), n=(48, 56, 48), shapes=np.zeros((0, 9)),
                             omega=1.0)
KINDS = ["plain", "ramp", "spikes", "exponents", "components"]


@pytest.fixture(scope="module")
def fc():
    from paper_2403_11636_gb300 import fc as m
    return m


def field(p, kind):
    nd, nn = p.dim + 1, [k + 1 for k in p.n]
    v = inputs.uniform_array(int(np.prod(nn)) * nd, 11).reshape(-1, nd)
    u = inputs.uniform_array(len(v), 12, 0.0, 1.0)
    ix = np.arange(len(v)) % nn[0]
    if kind == "ramp":
        v = v * (2.0 ** (-1.5 * ix))[:, None]
    elif kind == "spikes":
        v = v * np.where(u < 0.002, 1.0, 2.0 ** -40)[:, None]
    elif kind == "exponents":
        v = v * 2.0 ** (-60.0 * inputs.uniform_array(v.size, 13, 0.0, 1.0).reshape(v.shape))
    elif kind == "components":
        v = v * 2.0 ** -np.array([0.0, 30.0, 50.0, 60.0])[:nd]
    return np.ascontiguousarray(v.reshape(-1))


def nodes(p, count):
    """`count` nodes at least four layers from the faces, and their strides."""
    nn = [k + 1 for k in p.n]
    at, stride = 0, 1
    for k, n in enumerate(nn):
        at = at + stride * (4 + (inputs.uniform_array(count, 20 + k, 0.0, 1.0) * (n - 8)).astype(np.int64))
        stride *= n
    return at, [1, nn[0], nn[0] * nn[1]][:p.dim]


def box(dim, r):
    o = np.stack(np.meshgrid(*[np.arange(-r, r + 1)] * dim, indexing="ij"), -1).reshape(-1, dim)
    return o[:, ::-1]                                # x fastest


def check(y, at, nd, w, dof, v, terms):
    """w [nd, slots], dof [nodes, slots]: |y - w v| <= terms 2^-53 |w| |v| for every row."""
    wl, vl = w.astype(np.longdouble), v.astype(np.longdouble)[dof]
    for r in range(nd):
        want, size = (wl[r] * vl).sum(1), (abs(wl[r]) * abs(vl)).sum(1)
        off = abs(y[nd * at + r].astype(np.longdouble) - want)
        # (below 2^-1000 the products themselves are rounded as subnormals)
        worst = np.max(np.where(size > 2.0 ** -900, off / np.maximum(size, np.longdouble(2.0) ** -900), 0.0))
        assert float(worst) <= terms * 2.0 ** -53, (r, float(worst) * 2.0 ** 53)


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("dim", [2, 3])
def test_patch_rows(fc, dim, kind):
    """x = 0, so the sweep meets b itself and returns y = Inv b (omega = 1)."""
    p, nd = (EMPTY2, 3) if dim == 2 else (EMPTY3, 4)
    s = fc.Solver(p)
    b = field(p, kind)
    y = s.smooth(np.zeros_like(b), b).cpu().numpy()
    at, stride = nodes(p, 4000 if dim == 2 else 1500)
    w = s.patch_rows(int(at[0]))
    vel, prs = box(dim, 2) @ stride, box(dim, 1) @ stride
    off = np.concatenate([(vel[:, None] * nd + np.arange(dim)).reshape(-1), prs * nd + dim])
    check(y, at, nd, w, nd * at[:, None] + off, b, 18 if dim == 2 else 55)


@pytest.mark.parametrize("kind", KINDS)
def test_operator(fc, kind):
    p, nd = LARGE2, 3
    s = fc.Solver(p)
    x = field(p, kind)
    y = s.apply(x).cpu().numpy()
    at, stride = nodes(p, 20000)
    off, mid = box(2, 1) @ stride, int(at[0])
    w = np.zeros((nd, len(off), nd))                  # the rows of node mid, column by column
    for c in range(nd):
        for k, o in enumerate(off):
            e = np.zeros_like(x)
            e[nd * (mid + o) + c] = 1.0
            w[:, k, c] = s.apply(e).cpu().numpy()[nd * mid:nd * mid + nd]
    dof = nd * (at[:, None] + off)[:, :, None] + np.arange(nd)
    check(y, at, nd, w.reshape(nd, -1), dof.reshape(len(at), -1), x, 15)
