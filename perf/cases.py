"""The work a user of this library has it do, as cases with their inputs.

A pass is one window of a matrix sequence (Sec. V of the paper): the first matrix
is factored, every further one of the same pattern is refactored, and each is
solved for its right-hand sides, as a transient or power-flow simulation does
between two topology changes and as the serving loop does for a pattern's
requests.  Every pass starts with the factorization, so each pass has the same
history.  ``solve`` cases solve with factors made beforehand; ``host`` cases go
through the call that takes and returns host arrays.

Patterns depend on the case alone and are kept (a program analyses its pattern
once); values, solutions and right-hand sides depend on the seed.  Right-hand
sides are A x for a drawn x, so x is the value ``exact`` gives.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1601_05725_gb300 import basker, inputs

#: Refactorization values are the pattern's base values times (1 + N(0, SIGMA)).
SIGMA = 0.05


def listed():
    return [
        # the smallest call: one right-hand side of a 2,000-row circuit, factors at hand
        dict(name="circuit_solve", family="circuit", size=2000, mode="solve", steps=1, nrhs=1, precision=0),
        # a small circuit's time steps: BTF blocks around a four-leaf netlist, launch-bound
        dict(name="circuit_window", family="circuit", size=2000, mode="window", steps=4, nrhs=1, precision=0),
        # a small power grid of odd width, plain FP64
        dict(name="grid_small_window", family="grid", size=61, mode="window", steps=4, nrhs=1, precision=0),
        # the benchmark's power grid, FP64 factors with refined solves (its headline form)
        dict(name="grid_window", family="grid", size=316, mode="window", steps=4, nrhs=1, precision=2),
        # a mid-size grid in FP32 with FP64 refinement
        dict(name="grid_fp32_window", family="grid", size=149, mode="window", steps=4, nrhs=1, precision=1),
        # several load vectors on the benchmark's grid, factors at hand
        dict(name="grid_solve_many", family="grid", size=316, mode="solve", steps=1, nrhs=8, precision=0),
        # the end-to-end call on host arrays, a mid-size grid
        dict(name="grid_host_window", family="grid", size=120, mode="host", steps=4, nrhs=1, precision=0),
        # many independent circuits of 4 to 1,024 rows in one system, factored afresh for each set of values
        dict(name="blocks_factor", family="blocks", size=4096, mode="factor", steps=1, nrhs=1, precision=0),
        # a few hundred independent circuits over some time steps
        dict(name="blocks_small_window", family="blocks", size=301, mode="window", steps=3, nrhs=1, precision=0),
        # a served netlist of the middle of the serving range
        dict(name="netlist_window", family="netlist", size=20011, mode="window", steps=4, nrhs=1, precision=0),
        # a large served netlist, whose repivoting dominates the serving loop
        dict(name="netlist_large_window", family="netlist", size=150001, mode="window", steps=2, nrhs=1, precision=0),
        # a circuit with supply rails and many BTF blocks, four right-hand sides
        dict(name="rails_window", family="rails", size=100003, mode="window", steps=2, nrhs=4, precision=0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


#: Sizes of each family: rows, grid width or number of blocks.
RANGES = {"circuit": (300, 30000), "grid": (24, 316), "blocks": (64, 4096), "netlist": (5000, 150000),
          "rails": (20000, 100000)}


def draw(rng):
    """One more case of the same ranges."""
    family = rng.choice(["circuit", "grid", "grid", "blocks", "netlist", "netlist", "rails"])
    size = _log_int(rng, *RANGES[family])
    mode = rng.choice(["window", "window", "window", "solve", "host", "factor"])
    steps = 1 if mode in ("solve", "factor") else rng.randint(2, 4 if size < 50000 else 2)
    return dict(family=family, size=size, mode=mode, steps=steps, nrhs=rng.choice([1, 1, 1, 2, 3, 4, 8]),
                precision=rng.choice([0, 0, 0, 1, 2]))


def _tiled_blocks(count):
    """``count`` independent netlist blocks: up to 512 distinct ones, repeated
    (their values differ: every entry is drawn anew for each seed)."""
    base = inputs.block_diagonal_problem(3003, nblocks=min(count, 512), name="blocks")
    reps = -(-count // 512)
    if reps == 1:
        return base
    keep = count - 512 * (reps - 1)              # blocks of the last, partial copy
    n, nnz = base.n, base.nnz
    # B's order is the block order, so a partial copy is a leading part of B; A is
    # kept unscrambled between the copies (each copy carries its own scramble)
    full = reps - 1
    colptr = np.concatenate([base.colptr[:-1].astype(np.int64) + k * nnz for k in range(full)] + [[full * nnz]])
    rowind = np.concatenate([base.rowind + k * n for k in range(full)])
    P = np.concatenate([base.P + k * n for k in range(full)])
    Q = np.concatenate([base.Q + k * n for k in range(full)])
    bptr = np.concatenate([base.block_ptr[:-1] + k * n for k in range(full)] + [[full * n]])
    values = np.tile(base.values, full)
    if keep:
        tail = base if keep == 512 else inputs.block_diagonal_problem(3004, nblocks=keep, name="blocks")
        colptr = np.concatenate([colptr[:-1], tail.colptr.astype(np.int64) + full * nnz])
        rowind = np.concatenate([rowind, tail.rowind + full * n])
        P = np.concatenate([P, tail.P + full * n])
        Q = np.concatenate([Q, tail.Q + full * n])
        bptr = np.concatenate([bptr[:-1], tail.block_ptr + full * n])
        values = np.concatenate([values, tail.values])
    i32 = functools.partial(np.ascontiguousarray, dtype=np.int32)
    return inputs.Problem(name="blocks", n=int(bptr[-1]), colptr=i32(colptr), rowind=i32(rowind), values=values,
                          P=i32(P), Q=i32(Q), block_ptr=i32(bptr), meta=dict(seed=3003))


@functools.lru_cache(maxsize=None)
def _problem(family, size):
    """The pattern (and base values) of a case."""
    if family == "circuit":                      # 40 % of the rows in blocks of one or two rows
        small = int(round(0.4 * size))
        return inputs.netlist_problem(3001, n_small=small, small_sizes=(1, 2), m_netlist=size - small, depth=2)
    if family == "grid":
        return inputs.grid_problem(3002, k=size, depth=min(4, max(2, round(math.log2(size / 20)))))
    if family == "blocks":
        return _tiled_blocks(size)
    if family == "netlist":                      # the serving stream's patterns
        return inputs.netlist_problem(3005, n_small=0, m_netlist=size,
                                      depth=min(5, max(2, round(math.log2(size / 2000)))))
    if family == "rails":                        # the two-million-row circuit's structure, scaled down
        return inputs.config4(3006, n=size, n_rails=max(4, size // 10000),
                              rail_deg=(size // 2000, size // 40))
    raise ValueError(family)


@functools.lru_cache(maxsize=None)
def _columns(family, size):
    p = _problem(family, size)
    return np.repeat(np.arange(p.n), np.diff(p.colptr))


def _draws(case, seed):
    """Per step: values of A, the solution X (n, nrhs) and B = A X."""
    p, cols = _problem(case["family"], case["size"]), _columns(case["family"], case["size"])
    rng = np.random.default_rng([seed & 0x7fffffff, 17])
    out = []
    for _ in range(case["steps"]):
        v = p.values * (1.0 + SIGMA * rng.standard_normal(p.nnz))
        x = rng.standard_normal((p.n, case["nrhs"]))
        b = np.stack([np.bincount(p.rowind, weights=v * x[cols, q], minlength=p.n) for q in range(case["nrhs"])], 1)
        out.append((v, x, b))
    return out


def prepare(case, seed):
    p = _problem(case["family"], case["size"])
    h = basker.Handle.from_problem(p, precision=case["precision"])
    one = case["nrhs"] == 1
    steps = [(v, b[:, 0] if one else b) for v, _, b in _draws(case, seed)]
    if case["mode"] == "host":
        return dict(case=case, handle=h, steps=steps)
    # right-hand sides column-major, as the solve takes them
    dev = [(torch.as_tensor(v, device="cuda"),
            torch.as_tensor(b, device="cuda") if one else
            torch.as_tensor(np.ascontiguousarray(b.T), device="cuda").t()) for v, b in steps]
    if case["mode"] == "solve":
        h.factor(dev[0][0])
    return dict(case=case, handle=h, steps=dev)


def run(state):
    h, mode = state["handle"], state["case"]["mode"]
    if mode == "host":
        # a long-lived handle: the call refactors along the sequence
        return [h.refactor_solve_host(v, b) for v, b in state["steps"]]
    out = []
    for k, (v, b) in enumerate(state["steps"]):
        if mode != "solve":
            if k == 0:
                h.factor(v)
            else:
                h.refactor(v)
        out.append(h.solve(b))
    return out


@functools.lru_cache(maxsize=None)
def _counts(family, size):
    lc, uc = basker.symbolic_counts(_problem(family, size))
    lc, uc = lc.astype(np.float64), uc.astype(np.float64)
    # the pattern is nearly symmetric: row j of U holds about as many entries as L's column j
    return float(lc.sum()), float(uc.sum()), float((lc * (2 * lc + 1)).sum())


def work(case):
    """Per step: values read, factors written (values and indices) and read by the
    solve, right-hand sides read, solutions written; the factorization's and the
    solve's operations on the natural pivots' pattern."""
    p = _problem(case["family"], case["size"])
    nl, nu, fl = _counts(case["family"], case["size"])
    v = 4 if case["precision"] == 1 else 8
    solve_b = (v + 4) * (nl + nu) + 16 * p.n * case["nrhs"]
    solve_f = 2 * (nl + nu) * case["nrhs"]
    if case["mode"] == "solve":
        return {"bytes": solve_b, "flops": solve_f}
    return {"bytes": case["steps"] * (12 * p.nnz + (v + 4) * (nl + nu) + solve_b),
            "flops": case["steps"] * (fl + solve_f)}


def exact(case, seed):
    one = case["nrhs"] == 1
    return [x[:, 0] if one else x for _, x, _ in _draws(case, seed)]
