"""Separator columns of thousands of steps (supply rails): the reach with their
descendant nodes in parallel, and its hand-over of columns whose logs outgrow their
room, against the oracle bit for bit."""
import numpy as np
import pytest

import oracle
from paper_1601_05725_gb300 import basker, build
from paper_1601_05725_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _same(h, f):
    prow, L, U = h.export()
    np.testing.assert_array_equal(prow, f.prow)
    for a, b in ((L, f.L), (U, f.U)):
        np.testing.assert_array_equal(a.indptr, b.indptr)
        np.testing.assert_array_equal(a.indices, b.indices)
        np.testing.assert_array_equal(a.data, b.data)


@pytest.mark.parametrize("rails,deg,slack", [
    (4, (2500, 4000), 1.0),       # logs that fit
    (4, (2500, 4000), 0.0),       # U columns to the spill pool
    (24, (3000, 5500), 1.0),      # logs that do not
])
def test_rail_columns_match_oracle(rails, deg, slack):
    import torch
    build.build()
    basker.load()
    prob = I.config4(41, n=9000, n_rails=rails, rail_deg=deg)
    _, u = basker.symbolic_counts(prob)
    assert u.max() >= 2000, "no column of the size the test is for"
    o = oracle.OracleLU(prob)
    assert o.factor() == "OK"
    f = o.factors()
    h = basker.Handle.from_problem(prob, slack=slack)
    h.factor(torch.as_tensor(prob.values, device="cuda"))
    _same(h, f)
    for k in (1, 2):
        v = I.refactor_values(prob, k, sigma=0.2)
        assert o.factor(v, pref=f.prow) == "OK"
        f = o.factors()
        h.refactor(torch.as_tensor(v, device="cuda"))
        _same(h, f)
