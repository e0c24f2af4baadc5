"""Of several columns that fail, in a separator and in blocks behind the ND block, the
first is named, whichever path a call takes."""
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


def _failing(prob, v, columns):
    """v with zero columns of B (a NaN where the column is given as ~c)."""
    w = v.copy()
    for c in columns:
        q = prob.Q[c if c >= 0 else ~c]
        w[prob.colptr[q]:prob.colptr[q + 1]] = 0.0 if c >= 0 else np.nan
    return w


TREES = {
    "thin": dict(sizes=[300, 300, 4, 300, 300, 4, 5], chain=True),
    "dense": dict(sizes=[40, 40, 30, 40, 40, 30, 45], density=1.0),
}


def _make(tree):
    kw = dict(TREES[tree])
    prob = nd_problem(11, kw.pop("sizes"), before=[2], after=[3, 1, 4], **kw)
    ptr, n = prob.nd_node_ptr, prob.n
    return prob, [int(ptr[2]), int(ptr[6]) + 1], [n - 6, n - 1]


@pytest.mark.parametrize("tree", sorted(TREES))
@pytest.mark.parametrize("sep", [0, 1])          # a separator of level 1, the root
@pytest.mark.parametrize("nan", [False, True])
def test_factorization(tree, sep, nan):
    prob, seps, blocks = _make(tree)
    o = oracle.OracleLU(prob)
    h = basker.Handle.from_problem(prob)
    for _ in range(2):
        v = _failing(prob, prob.values, [~seps[sep] if nan else seps[sep]] + blocks)
        status = o.factor(v)
        assert status == ("NAN" if nan else "SINGULAR")
        with pytest.raises(basker.BaskerError) as e:
            h.factor(_dev(v))
        assert (e.value.name, e.value.column) == (status, o.info_col)
        assert o.factor() == "OK"
        h.factor(_dev(prob.values))
        _same(h, o.factors())


@pytest.mark.parametrize("tree", sorted(TREES))
@pytest.mark.parametrize("settled", [0, 3])      # the teams, or the stored patterns first
def test_refactorization(tree, settled):
    prob, seps, blocks = _make(tree)
    o = oracle.OracleLU(prob)
    for bad in ([seps[0]] + blocks, [~seps[1]] + blocks, blocks):
        h = basker.Handle.from_problem(prob)
        assert o.factor() == "OK"
        h.factor(_dev(prob.values))
        for _ in range(settled):
            assert o.factor(pref=o.factors().prow) == "OK"
            h.refactor(_dev(prob.values))
        v = _failing(prob, prob.values, bad)
        status = o.factor(v, pref=o.factors().prow)
        with pytest.raises(basker.BaskerError) as e:
            h.refactor(_dev(v))
        assert (e.value.name, e.value.column) == (status, o.info_col)
        assert o.factor() == "OK"
        h.factor(_dev(prob.values))
        _same(h, o.factors())


@pytest.mark.parametrize("tree", sorted(TREES))
@pytest.mark.parametrize("kw", [dict(refactor_switch=1), dict(refactor_switch=3), dict(factor_mode=1),
                                dict(factor_mode=1, refactor_switch=3)], ids=str)
def test_refactorization_without_teams(tree, kw):
    """Rounds, the one-block repair and the column-by-column in-node phase; failures among
    rejected pivots."""
    prob, seps, blocks = _make(tree)
    o = oracle.OracleLU(prob)
    ptr = prob.nd_node_ptr
    leaf = [int(ptr[0]) + 3, int(ptr[4]) + 2]
    for bad in ([seps[0]] + blocks, [~seps[1]] + blocks, [seps[1]] + leaf, leaf[::-1] + blocks):
        h = basker.Handle.from_problem(prob, **kw)
        assert o.factor() == "OK"
        h.factor(_dev(prob.values))
        v = _failing(prob, I.refactor_values(prob, 1, sigma=0.7), bad)
        status = o.factor(v, pref=o.factors().prow)
        assert status != "OK"
        with pytest.raises(basker.BaskerError) as e:
            h.refactor(_dev(v))
        assert (e.value.name, e.value.column) == (status, o.info_col)
        assert o.factor() == "OK"
        h.factor(_dev(prob.values))
        _same(h, o.factors())
