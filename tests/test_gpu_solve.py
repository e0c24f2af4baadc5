"""The solve's two forms (a job per ND leaf or run of BTF blocks; rows over the
whole GPU) against the oracle bit for bit, for one right-hand side, a lane group
that is not full, a full warp of them and one batch more."""
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


PROBLEMS = {
    # blocks in a chain around an ND block; runs of more than 1,024 rows of small blocks
    "chain": lambda: I.netlist_problem(31, n_small=2600, small_sizes=(1, 3), m_netlist=900, depth=2),
    # couplings to random later blocks, rails in the root separator (long rows)
    "rails": lambda: I.config4(32, n=9000, n_rails=6, rail_deg=(50, 900)),
    # no ND, no coupling
    "blocks": lambda: I.block_diagonal_problem(33, nblocks=150, size_range=(1, 700)),
    # dense columns: rows over the whole GPU; separators swept
    "grid": lambda: I.grid_problem(34, k=52, depth=3),
    # an ND tree of one leaf, and none
    "one_leaf": lambda: I.netlist_problem(35, n_small=30, m_netlist=400, depth=0),
}


@pytest.mark.parametrize("name", sorted(PROBLEMS))
@pytest.mark.parametrize("nrhs", [1, 2, 5, 32, 33])
def test_solve_matches_oracle(name, nrhs):
    import torch
    prob = PROBLEMS[name]()
    o = oracle.OracleLU(prob)
    assert o.factor() == "OK"
    h = basker.Handle.from_problem(prob)
    h.factor(torch.as_tensor(prob.values, device="cuda"))
    rng = np.random.default_rng(nrhs)
    for _ in range(2):            # the second solve starts from the first one's buffers
        B = rng.standard_normal((prob.n, nrhs))
        X = h.solve(torch.as_tensor(B, device="cuda")).cpu().numpy()
        np.testing.assert_array_equal(X, o.solve(B).reshape(prob.n, nrhs))


@pytest.mark.parametrize("name", ["chain", "grid"])
def test_solve_carries_non_finite_right_hand_sides(name):
    """Infinities and NaN (also the one whose bits mark a missing value) end in the
    solution, and the call returns."""
    import torch
    prob = PROBLEMS[name]()
    o = oracle.OracleLU(prob)
    assert o.factor() == "OK"
    h = basker.Handle.from_problem(prob)
    h.factor(torch.as_tensor(prob.values, device="cuda"))
    b = np.random.default_rng(3).standard_normal(prob.n)
    b[[5, prob.n // 2]] = np.inf, np.nan
    b.view(np.uint64)[prob.n - 7] = np.uint64(0xFFFFFFFFFFFFFFFF)
    x, xo = h.solve(torch.as_tensor(b, device="cuda")).cpu().numpy(), o.solve(b)
    np.testing.assert_array_equal(x, xo)          # NaN equal to NaN


@pytest.mark.parametrize("m,nrhs", [(1025, 1), (1100, 3), (481, 32), (500, 33)])
def test_separators_swept_in_place(m, nrhs):
    """A separator with more values than a sweeper's shared memory holds (1,024 rows; 480
    with 32 right-hand sides) is swept in global memory."""
    import torch
    prob = nd_problem(m, [7, 5, m], density=0.02)
    o = oracle.OracleLU(prob)
    assert o.factor() == "OK"
    h = basker.Handle.from_problem(prob)
    h.factor(torch.as_tensor(prob.values, device="cuda"))
    rng = np.random.default_rng(nrhs)
    for _ in range(3):
        B = rng.standard_normal((prob.n, nrhs))
        X = h.solve(torch.as_tensor(B, device="cuda")).cpu().numpy()
        np.testing.assert_array_equal(X, o.solve(B).reshape(prob.n, nrhs))
