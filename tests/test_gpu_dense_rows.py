"""Separators eliminated with their rows dealt over one block, a cluster of blocks, or
(too large for either) with their columns dealt over a cluster: sizes around the edges
of the three, against the oracle bit for bit, and in FP32 against the column-by-column
elimination."""
import numpy as np
import pytest

import oracle
from paper_1601_05725_gb300 import basker, build
from paper_1601_05725_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def _problem(seed, a, m, p, leaf=5):
    """Four leaves of `leaf` unknowns, two separators of a, a root of m: each node's block
    random at density p (the leaves' a chain), each separator tied to the nodes below it."""
    rng = np.random.default_rng(seed)
    sizes = [leaf, leaf, a, leaf, leaf, a, m]
    ptr = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32)
    n = int(ptr[-1])
    D = np.zeros((n, n))
    span = [slice(ptr[i], ptr[i + 1]) for i in range(7)]

    def fill(r, c, density):
        shape = (r.stop - r.start, c.stop - c.start)
        v = rng.uniform(-1, 1, shape) * (rng.random(shape) < density)
        D[r, c] = np.where(v != 0, v, D[r, c])

    for i in (0, 1, 3, 4):
        for k in range(int(ptr[i]), int(ptr[i + 1]) - 1):
            D[k, k + 1], D[k + 1, k] = rng.uniform(-1, 1, 2)
    for i in (2, 5, 6):
        fill(span[i], span[i], p)
    for s, below in ((2, (0, 1)), (5, (3, 4)), (6, (0, 1, 2, 3, 4, 5))):
        for b in below:
            d = min(1.0, 8.0 / max(sizes[s], sizes[b]))
            fill(span[s], span[b], d)
            fill(span[b], span[s], d)
    D[np.arange(n), np.arange(n)] = rng.uniform(0.5, 1.0, n)
    cols, rows = np.nonzero(D.T)
    colptr = np.concatenate([[0], np.cumsum(np.bincount(cols, minlength=n))]).astype(np.int32)
    eye = np.arange(n, dtype=np.int32)
    return I.Problem("separators", n, colptr, rows.astype(np.int32), np.ascontiguousarray(D.T[cols, rows]), eye, eye.copy(),
                     np.array([0, n], np.int32), 0, 4, ptr)


def _same(h, f):
    prow, L, U = h.export()
    np.testing.assert_array_equal(prow, f.prow)
    for x, y in ((L, f.L), (U, f.U)):
        np.testing.assert_array_equal(x.indptr, y.indptr)
        np.testing.assert_array_equal(x.indices, y.indices)
        np.testing.assert_array_equal(x.data, y.data)


@pytest.mark.parametrize("a,m,p", [
    (1, 1, 1.0),
    (31, 33, 0.3),
    (63, 64, 0.5),
    (64, 65, 0.2),
    (60, 300, 0.1),       # one block, more rows than threads that divide
    (65, 150, 1.0),
    (70, 1000, 0.02),     # 134 rows a block; a root too large for the rows of a cluster
])
def test_separator_sizes_match_oracle(a, m, p):
    import torch
    build.build()
    basker.load()
    prob = _problem(a + m, a, m, p)
    dev = lambda v: torch.as_tensor(v, device="cuda")
    for tau in (1e-3, 1.0):
        o = oracle.OracleLU(prob)
        assert o.factor(tau=tau) == "OK"
        f = o.factors()
        h = basker.Handle.from_problem(prob, tau=tau)
        h.factor(dev(prob.values))
        assert h.info()["kernel_calls"]["dense_node"] > 0
        _same(h, f)
        v = I.refactor_values(prob, 1, sigma=0.5)
        assert o.factor(v, tau=tau, pref=f.prow) == "OK"
        h.refactor(dev(v))
        _same(h, o.factors())
    single = []
    for mode in (0, 1):
        h = basker.Handle.from_problem(prob, factor_mode=mode, precision=1)
        h.factor(dev(prob.values))
        single.append(h.export())
    np.testing.assert_array_equal(single[0][0], single[1][0])
    for x, y in zip(single[0][1:], single[1][1:]):
        np.testing.assert_array_equal(x.indptr, y.indptr)
        np.testing.assert_array_equal(x.indices, y.indices)
        np.testing.assert_array_equal(x.data, y.data)
