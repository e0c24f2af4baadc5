"""ND separators whose descendants are all empty, which are factored and solved as leaves,
against the oracle bit for bit."""
import numpy as np
import pytest

import oracle
from paper_1601_05725_gb300 import basker, build
from paper_1601_05725_gb300 import inputs as I
from tests.nd_cases import EMPTY, nd_problem

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


def sequence_matches_oracle(prob, steps, **kw):
    """A factorization, ``steps`` refactorizations and solves of 1 and 3 right-hand sides."""
    rng = np.random.default_rng(1)
    o = oracle.OracleLU(prob)
    h = basker.Handle.from_problem(prob, **kw)
    f = None
    for k in range(steps + 1):
        v = I.refactor_values(prob, k, sigma=0.4) if k else prob.values
        assert o.factor(v, pref=f.prow if k else None) == "OK"
        f = o.factors()
        (h.refactor if k else h.factor)(_dev(v))
        _same(h, f)
        for nrhs in (1, 3):
            B = rng.standard_normal((prob.n, nrhs))
            np.testing.assert_array_equal(h.solve(_dev(B)).cpu().numpy(), o.solve(B).reshape(prob.n, nrhs))
    return h


@pytest.mark.parametrize("switch", [0, 1, 2, 3])
@pytest.mark.parametrize("name", sorted(EMPTY))
def test_empty_descendants_match_oracle(name, switch):
    sizes, kw = EMPTY[name]
    sequence_matches_oracle(nd_problem(5, sizes, **kw), 3, refactor_switch=switch)


@pytest.mark.parametrize("sizes", [
    [300, 300, 0, 300, 300, 0, 3],
    [200, 0, 0, 150, 0, 0, 2, 100, 130, 0, 120, 110, 0, 4, 5],       # the same below two levels of separators
    [300, 300, 2, 300, 300, 0, 3],                                   # rows in one of them
])
@pytest.mark.parametrize("precision", [0, 1])
def test_separators_in_stages_above_an_empty_level(sizes, precision):
    """No separator of level 1 has rows: the leaves' part of the columns above goes
    ahead all the same."""
    prob = nd_problem(5, sizes, chain=True)
    _, u = basker.symbolic_counts(prob)
    assert u.max() >= 128, "no column of the size that goes in stages"
    if precision == 0:
        sequence_matches_oracle(prob, 2)
        return
    # FP32 factors: the stages against the column-by-column form
    out = []
    for mode in (0, 1):
        h = basker.Handle.from_problem(prob, precision=1, factor_mode=mode)
        h.factor(_dev(prob.values))
        h.refactor(_dev(I.refactor_values(prob, 1, sigma=0.4)))
        out.append(h.export())
    np.testing.assert_array_equal(out[0][0], out[1][0])
    for a, b in zip(out[0][1:], out[1][1:]):
        np.testing.assert_array_equal(a.indptr, b.indptr)
        np.testing.assert_array_equal(a.indices, b.indices)
        np.testing.assert_array_equal(a.data, b.data)
