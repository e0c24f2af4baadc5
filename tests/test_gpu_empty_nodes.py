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
