"""A refactorization whose wait gave up (a one-cycle budget): its half-new factors solve
nothing, the next refactorization or factorization gives the oracle's."""
import numpy as np
import pytest

import oracle
from paper_1601_05725_gb300 import basker, build
from paper_1601_05725_gb300 import inputs as I
from tests.nd_cases import nd_problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    basker.load()


def _dev(v):
    import torch
    return torch.as_tensor(v, device="cuda")


def _same(h, f):
    prow, L, U = h.export()
    np.testing.assert_array_equal(prow, f.prow)
    for a, b in ((L, f.L), (U, f.U)):
        np.testing.assert_array_equal(a.indptr, b.indptr)
        np.testing.assert_array_equal(a.indices, b.indices)
        np.testing.assert_array_equal(a.data, b.data)


def _times_out(prob, v, **kw):
    """A handle whose refactorization of v has given up (the waits' luck may take a few)."""
    for _ in range(5):
        h = basker.Handle.from_problem(prob, wait_budget_cycles=1, **kw)
        h.factor(_dev(prob.values))
        try:
            h.refactor(_dev(v))
        except basker.BaskerError as e:
            assert e.name == "TIMEOUT"
            return h
        h.free()
    pytest.fail("no wait of the refactorization gave up")


def _refused(call):
    with pytest.raises(basker.BaskerError) as e:
        call()
    assert e.value.name == "NOT_FACTORED"


@pytest.mark.parametrize("make", [
    lambda: I.grid_problem(41, k=40, depth=3),
    lambda: I.netlist_problem(42, n_small=30, m_netlist=3000, depth=2),
])
@pytest.mark.parametrize("switch", [0, 1, 3])
def test_after_a_wait_that_gave_up(make, switch):
    prob = make()
    v = I.refactor_values(prob, 1, sigma=0.2)
    o = oracle.OracleLU(prob)
    assert o.factor() == "OK"
    pref = o.factors().prow
    h = _times_out(prob, v, refactor_switch=switch)
    b = _dev(np.ones(prob.n))
    _refused(lambda: h.solve(b))
    _refused(h.export)
    if switch:
        # one complete pass, which waits for nothing, from the pivots of before
        assert o.factor(v, pref=pref) == "OK"
        h.refactor(_dev(v))
        _same(h, o.factors())
    else:
        try:
            h.refactor(_dev(v))          # accepted; teams wait as well
        except basker.BaskerError as e:
            assert e.name == "TIMEOUT"
            _refused(lambda: h.solve(b))
    assert o.factor() == "OK"
    h.factor(_dev(prob.values))
    _same(h, o.factors())


@pytest.mark.parametrize("m", [40, 100])         # one block, a cluster of blocks
@pytest.mark.parametrize("switch", [0, 1, 3])
def test_budget_of_the_separators_elimination(m, switch):
    """Leaves of one row wait for nothing: only the elimination's messages do.  The budget
    is theirs too, and a factorization falls back on a pass that gives them their time."""
    prob = nd_problem(3, [1, 1, m])
    o = oracle.OracleLU(prob)
    assert o.factor() == "OK"
    f = o.factors()
    h = basker.Handle.from_problem(prob, wait_budget_cycles=1, refactor_switch=switch)
    for _ in range(2):
        h.factor(_dev(prob.values))
        _same(h, f)
        with pytest.raises(basker.BaskerError) as e:
            h.refactor(_dev(prob.values))
        assert e.value.name == "TIMEOUT"
        _refused(lambda: h.solve(_dev(np.ones(prob.n))))
    h = basker.Handle.from_problem(prob, refactor_switch=switch)
    h.factor(_dev(prob.values))
    h.refactor(_dev(prob.values))
    _same(h, f)
