"""The team factorization of ND leaves and BTF blocks (several warps a task, the
columns deciding in order) against the oracle, bit for bit, at the sizes where
its layouts change: teams of one, four, eight and sixteen warps, patterns of 32,
64 and 1,024 rows, x in shared memory or in the workspace; and its repair of a
stored-pattern pass."""
import numpy as np
import pytest

import oracle
from paper_1601_05725_gb300 import basker, build
from paper_1601_05725_gb300 import inputs as I
from tests import helpers as H

pytestmark = pytest.mark.gpu


def _dev(a):
    import torch
    return torch.as_tensor(a, device="cuda")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build()
    basker.load()


def _random_blocks(seed, sizes, per_col):
    """Independent unsymmetric blocks: a random diagonal of the off-diagonals' size
    and per_col random entries a column, so that many natural pivots are rejected."""
    import scipy.sparse as sp
    rng = np.random.default_rng(seed)
    mats = []
    for m in sizes:
        k = min(m, per_col)
        r = np.concatenate([rng.permutation(m)[:k] for _ in range(m)])
        M = sp.csc_matrix((rng.standard_normal(r.size), (r, np.repeat(np.arange(m), k))), shape=(m, m))
        mats.append(M + sp.diags(rng.uniform(0.05, 1.0, m)))
    return H.make_problem(sp.block_diag(mats), block_ptr=np.concatenate([[0], np.cumsum(sizes)]), scramble_seed=seed)


def _same(h, f):
    prow, L, U = h.export()
    np.testing.assert_array_equal(prow, f.prow)
    for a, b in ((L, f.L), (U, f.U)):
        np.testing.assert_array_equal(a.indptr, b.indptr)
        np.testing.assert_array_equal(a.indices, b.indices)
        np.testing.assert_array_equal(a.data, b.data)


def _sequence(prob, tau, steps, sigma, **kw):
    o = oracle.OracleLU(prob)
    assert o.factor(tau=tau) == "OK"
    f = o.factors()
    h = basker.Handle.from_problem(prob, tau=tau, **kw)
    h.factor(_dev(prob.values))
    _same(h, f)
    moved = 0
    for k in range(1, steps + 1):
        v = I.refactor_values(prob, k, sigma=sigma)
        assert o.factor(v, tau=tau, pref=f.prow) == "OK"
        g = o.factors()
        moved += int((g.prow != f.prow).sum())
        f = g
        h.refactor(_dev(v))
        _same(h, f)
        b = I.rhs_ones(prob, v)
        np.testing.assert_array_equal(h.solve(_dev(b)).cpu().numpy(), o.solve(b))
    return h, moved


@pytest.mark.parametrize("sizes,per_col", [
    ([1, 2, 15, 16, 17, 31, 32, 33], 3),                  # one warp up to 16 rows, then sixteen
    ([63, 64, 65, 97, 128], 2),                           # patterns around 32 and 64 rows
    ([5] * 40 + [40] * 400, 3),                           # eight warps a task
    ([24] * 1300, 3),                                     # four warps a task
    ([1023, 1024, 1025], 2),
    ([1300], 40),                                         # patterns past the listed 1,024 rows
])
def test_blocks_of_all_team_sizes(sizes, per_col):
    _, moved = _sequence(_random_blocks(7, sizes, per_col), 0.3, 2, 0.5)
    assert moved > 0


def test_leaves_with_x_in_the_workspace_and_spills():
    # leaves of about 1,900 rows (x does not fit on chip for sixteen warps), slack 0:
    # columns move to the spill pools
    prob = I.netlist_problem(19, n_small=0, m_netlist=7700, depth=2)
    _, moved = _sequence(prob, 1e-3, 2, 0.3, slack=0.0)
    assert moved > 0


@pytest.mark.parametrize("k,sigma", [(40, 0.05), (61, 0.1), (75, 0.08)])
def test_repair_of_a_stored_pattern_pass(k, sigma):
    prob = I.grid_problem(5, k=k, depth=2)
    h, moved = _sequence(prob, 1e-2, 4, sigma)
    assert moved > 0, "no pivot was rejected: the repair was not exercised"
    assert h.info()["kernel_calls"]["refactor_rounds"] > 0


def test_fp32_repair_equals_rounds():
    prob = I.grid_problem(6, k=48, depth=2)
    out = []
    for switch in (0, 1):
        h = basker.Handle.from_problem(prob, tau=1e-2, precision=1, refactor_switch=switch)
        h.factor(_dev(prob.values))
        for k in (1, 2, 3):
            h.refactor(_dev(I.refactor_values(prob, k, sigma=0.1)))
        out.append(h.export())
    np.testing.assert_array_equal(out[0][0], out[1][0])
    for a, b in zip(out[0][1:], out[1][1:]):
        np.testing.assert_array_equal(a.indptr, b.indptr)
        np.testing.assert_array_equal(a.indices, b.indices)
        np.testing.assert_array_equal(a.data, b.data)


def test_stored_patterns_serve_again_after_a_jump():
    """After one refactorization that rejects many pivots, a sequence that repeats is
    back on the stored patterns; the factors are the oracle's throughout."""
    prob = I.grid_problem(5, k=61, depth=2)
    o = oracle.OracleLU(prob)
    assert o.factor(tau=0.3) == "OK"
    f = o.factors()
    h = basker.Handle.from_problem(prob, tau=0.3)
    h.factor(_dev(prob.values))
    stored = []
    for k, sigma in ((1, 0.05), (1, 0.05), (1, 0.05), (2, 1.0), (2, 1.0), (2, 1.0)):
        v = I.refactor_values(prob, k, sigma=sigma)
        assert o.factor(v, tau=0.3, pref=f.prow) == "OK"
        f = o.factors()
        h.info()
        h.refactor(_dev(v))
        stored.append(h.info()["kernel_calls"]["static_refactor"])
        _same(h, f)
    assert stored == [1, 0, 1, 1, 0, 1]
