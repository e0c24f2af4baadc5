"""Separator columns in stages (their leaves first, all levels at once) and whole (one
level of separators, supply rails), against the oracle bit for bit; a factorization that
fails between the stages leaves the handle usable."""
import numpy as np
import pytest

import oracle
from paper_1601_05725_gb300 import basker, build
from paper_1601_05725_gb300 import inputs as I

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


@pytest.mark.parametrize("m,depth,rails", [
    (20000, 2, 0),
    (30000, 4, 0),
    (20000, 3, 5),     # rails in the root, behind two levels of separators
    (6000, 1, 5),      # one level: whole columns
])
def test_separator_columns_match_oracle(m, depth, rails):
    kw = dict(n_rails=rails, rail_deg=(2200, 4000)) if rails else {}
    prob = I.netlist_problem(90 + depth, n_small=40, m_netlist=m, depth=depth, **kw)
    _, u = basker.symbolic_counts(prob)
    root = u[prob.nd_node_ptr[-2]:prob.nd_node_ptr[-1]]
    assert root.max() >= (128 if depth > 1 else 2000), "no column of the size the test is for"
    o = oracle.OracleLU(prob)
    assert o.factor() == "OK"
    f = o.factors()
    h = basker.Handle.from_problem(prob)
    h.factor(_dev(prob.values))
    _same(h, f)
    for k in (1, 2):
        v = I.refactor_values(prob, k, sigma=0.3)
        assert o.factor(v, pref=f.prow) == "OK"
        f = o.factors()
        h.refactor(_dev(v))
        _same(h, f)


@pytest.mark.parametrize("node", [0, 2, 5])      # a leaf, separators of levels 1
def test_failure_between_the_stages(node):
    prob = I.netlist_problem(92, n_small=0, m_netlist=20000, depth=2)
    o = oracle.OracleLU(prob)
    h = basker.Handle.from_problem(prob)
    v = prob.values.copy()
    j = int(prob.nd_node_ptr[node])
    q = prob.Q[j]
    v[prob.colptr[q]:prob.colptr[q + 1]] = 0.0
    assert o.factor(v) == "SINGULAR"
    with pytest.raises(basker.BaskerError) as e:
        h.factor(_dev(v))
    assert e.value.name == "SINGULAR" and e.value.column == o.info_col
    assert o.factor(prob.values) == "OK"
    h.factor(_dev(prob.values))
    _same(h, o.factors())


@pytest.mark.parametrize("make", [
    lambda: I.netlist_problem(94, n_small=60, m_netlist=20000, depth=2),
    lambda: I.config4(95, n=9000, n_rails=4, rail_deg=(2500, 4000)),
    lambda: I.block_diagonal_problem(96, nblocks=60, size_range=(1, 500)),
])
def test_sequence_that_settles_and_moves_again(make):
    """Values repeated until no pivot moves (the stored patterns serve), then new ones."""
    prob = make()
    o = oracle.OracleLU(prob)
    assert o.factor() == "OK"
    f = o.factors()
    h = basker.Handle.from_problem(prob)
    h.factor(_dev(prob.values))
    static = 0
    for k in (1, 1, 1, 2, 2, 2, 1):
        v = I.refactor_values(prob, k, sigma=0.3)
        assert o.factor(v, pref=f.prow) == "OK"
        f = o.factors()
        h.info()
        h.refactor(_dev(v))
        static += h.info()["kernel_calls"]["static_refactor"]
        _same(h, f)
    assert static > 0, "no refactorization on the stored patterns"
