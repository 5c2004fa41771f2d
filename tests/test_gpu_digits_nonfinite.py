"""An infinity or NaN in a tile of class products reaches exactly the rows whose
products read it, as in the general kernels: the operator couples a velocity
component to itself and the pressure, a patch row reads every slot of its box.
The other rows are as without it (bounds of test_gpu_digits.py)."""
import numpy as np
import pytest

from paper_2403_11636_gb300 import inputs
from tests.gpu_util import rel
from tests.test_gpu_digits import OPER_TOL, PROBS, PROBS3, square

pytestmark = pytest.mark.gpu
ALL = {**PROBS, **PROBS3,
       "800x640": square(800, 640, nlevels=6), "open 800x640": square(800, 640, nlevels=6, preset=2)}


@pytest.fixture(scope="module")
def fc():
    from paper_2403_11636_gb300 import fc as m
    return m


def around(p, at, r):
    """Nodes of the (2 r + 1)^d box of node `at` (a tuple), as a mask."""
    m = np.zeros([k + 1 for k in reversed(p.n)], bool)
    m[tuple(slice(k - r, k + r + 1) for k in reversed(at))] = True
    return m.reshape(-1)


# a fluid node away from obstacle and walls
AT = {"384x352": (40, 300), "800x640": (80, 560), "open 800x640": (690, 90), "48": (4, 40, 6)}


@pytest.mark.parametrize("bad", [np.inf, np.nan])
@pytest.mark.parametrize("name", ["800x640", "open 800x640"])
def test_operator(fc, name, bad):
    p, nd = ALL[name], 3
    s = fc.Solver(p)
    x = inputs.random_vector(p, 9)
    ref = s.apply(x).cpu().numpy()
    i = AT[name][0] + (p.n[0] + 1) * AT[name][1]
    for c in range(nd):
        y = x.copy()
        y[nd * i + c] = bad
        got = s.apply(y).cpu().numpy()
        want = np.zeros((len(x) // nd, nd), bool)
        want[around(p, AT[name], 1)] = [c == 0 or c == 2, c == 1 or c == 2, True]
        want = want.reshape(-1)
        np.testing.assert_array_equal(~np.isfinite(got), want)
        assert rel(got[~want], ref[~want]) <= OPER_TOL


@pytest.mark.parametrize("bad", [np.inf, np.nan])
@pytest.mark.parametrize("name", ["384x352", "48"])
def test_sweep(fc, name, bad):
    p = ALL[name]
    nd = p.dim + 1
    s = fc.Solver(p)
    x, b = inputs.random_vector(p, 9), inputs.random_vector(p, 10)
    ref = s.smooth(x, b).cpu().numpy()
    i = sum(k * int(np.prod([n + 1 for n in p.n[:q]])) for q, k in enumerate(AT[name]))
    for c in (0, p.dim):
        y = b.copy()
        y[nd * i + c] = bad
        got = s.smooth(x, y).cpu().numpy()
        want = np.repeat(around(p, AT[name], 2 if c < p.dim else 1), nd)
        np.testing.assert_array_equal(~np.isfinite(got), want)
        assert rel(got[~want] - x[~want], ref[~want] - x[~want]) <= 1e-10
