"""The factors by rows, through the solves that read them: rows at the edges of each way
of ordering their entries, in one BTF block (columns far apart: compared with each other),
close together (a map over their range), and in a leaf whose row reaches into separators
behind a large leaf (a map over the leaf's rows and its ancestors')."""
import numpy as np
import pytest
import scipy.sparse as sp

import oracle
from paper_1601_05725_gb300 import basker, build
from paper_1601_05725_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _problem(where, length):
    """A diagonal, one row of U and one of L with `length` entries each."""
    rng = np.random.default_rng(length)
    leaf, big, sep = 40, 17000, 600
    n = leaf + big + sep
    if where == "leaf":
        up = leaf + big + rng.choice(sep, length, replace=False)
    elif where == "far":
        up = 2 + rng.choice(n - 4, length, replace=False)
        up[0], up[1] = 2, n - 2
        up = np.unique(up)
    else:
        up = 2 + rng.choice(900, length, replace=False)
    low = up if where != "leaf" else rng.choice(leaf + big - 2, length, replace=False)
    rows = np.concatenate([np.arange(n), np.zeros(up.size, int), np.full(low.size, n - 1)])
    cols = np.concatenate([np.arange(n), up, low])
    keep = (rows == cols) | ((cols != 0) & (cols != n - 1))
    rows, cols = rows[keep], cols[keep]
    vals = np.where(rows == cols, rng.uniform(2, 3, rows.size), rng.uniform(-1, 1, rows.size))
    A = sp.csc_matrix((vals, (rows, cols)), (n, n))
    A.sort_indices()
    eye = np.arange(n, dtype=np.int32)
    nd = (0, 2, np.array([0, leaf, leaf + big, n], np.int32)) if where == "leaf" else (-1, 0, np.zeros(0, np.int32))
    return I.Problem("rows", n, A.indptr.astype(np.int32), A.indices.astype(np.int32), A.data, eye, eye.copy(),
                     np.array([0, n], np.int32), *nd)


@pytest.mark.parametrize("where", ["near", "far", "leaf"])
@pytest.mark.parametrize("length", [3, 31, 32, 33, 34, 511, 512, 513])
def test_rows_of_all_lengths_solve_as_the_oracle(where, length):
    import torch
    build.build()
    basker.load()
    prob = _problem(where, length)
    o = oracle.OracleLU(prob)
    assert o.factor() == "OK"
    h = basker.Handle.from_problem(prob)
    h.factor(torch.as_tensor(prob.values, device="cuda"))
    # an order other than the oracle's shows in the sums' last bits
    b = np.random.default_rng(1).standard_normal(prob.n)
    np.testing.assert_array_equal(h.solve(torch.as_tensor(b, device="cuda")).cpu().numpy(), o.solve(b))
