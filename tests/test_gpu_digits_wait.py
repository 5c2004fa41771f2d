"""Tiles of class products whose wait for the tensor cores runs out
(FC_DIGIT_WAIT_NS=0): the products are formed in FP64, every node's once, with
no part of an unfinished one.  Bounds as in test_gpu_digits.py."""
import pytest

from oracle import oracle as O
from paper_2403_11636_gb300 import inputs
from tests.gpu_util import rel
from tests.test_gpu_digits import OPER_TOL, PROBS, PROBS3, SWEEP_TOL, fields, square

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fc():
    from paper_2403_11636_gb300 import fc as m
    return m


# several tiles in both directions, with an obstacle among them
@pytest.mark.parametrize("name", ["384x352", "528x272"])
def test_given_up_2d(fc, name, monkeypatch):
    monkeypatch.setenv("FC_DIGIT_WAIT_NS", "0")
    p = PROBS[name]
    L = O.Level.from_problem(p)
    A, b, _ = L.csr()
    s = fc.Solver(p)
    x = fields(L, "plain", 5)
    assert rel(s.apply(x).cpu().numpy(), A @ x) <= OPER_TOL
    assert rel(s.residual(x, b).cpu().numpy(), b - A @ x) <= OPER_TOL
    assert rel(s.smooth(x, b).cpu().numpy() - x, L.sweep(b, x) - x) <= SWEEP_TOL


def test_given_up_operator(fc, monkeypatch):
    p = square(800, 640, nlevels=6)
    s = fc.Solver(p)
    monkeypatch.setenv("FC_DIGIT_WAIT_NS", "0")
    t = fc.Solver(p)
    x, b = inputs.uniform_array(s.ndof(), 5), s.rhs()
    assert rel(t.apply(x).cpu().numpy(), s.apply(x).cpu().numpy()) <= OPER_TOL
    assert rel(t.residual(x, b).cpu().numpy(), s.residual(x, b).cpu().numpy()) <= OPER_TOL
    with pytest.raises(fc.FcError):
        t.sync()


@pytest.mark.parametrize("name", ["48", "pores"])
def test_given_up_3d(fc, name, monkeypatch):
    p = PROBS3[name]
    s = fc.Solver(p)
    monkeypatch.setenv("FC_DIGIT_WAIT_NS", "0")
    t = fc.Solver(p)
    x, b = inputs.uniform_array(s.ndof(), 5), inputs.uniform_array(s.ndof(), 7)
    want = s.smooth(x, b, nsweeps=2).cpu().numpy()
    assert rel(t.smooth(x, b, nsweeps=2).cpu().numpy() - x, want - x) <= 1e-11


@pytest.mark.parametrize("name", ["384x352", "48"])
def test_given_up_is_reported_once(fc, name, monkeypatch):
    p = {**PROBS, **PROBS3}[name]
    s = fc.Solver(p)
    monkeypatch.setenv("FC_DIGIT_WAIT_NS", "0")
    t = fc.Solver(p)
    x, b = inputs.uniform_array(s.ndof(), 5), inputs.uniform_array(s.ndof(), 7)
    t.sync()
    s.smooth(x, b)
    s.sync()
    for _ in range(2):
        t.smooth(x, b)
        with pytest.raises(fc.FcError) as e:
            t.sync()
        assert e.value.code == fc.FC_ERR_TIMEOUT
        t.sync()
