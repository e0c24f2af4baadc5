"""The solve's host-side plan (csrc/solve_plan.cpp): every row has one forward and one
backward item, as a job's or as a row of the separators, in every shape of ND tree; the
places of a leaf's job are those that the leaf order fills after a factorization."""
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_1601_05725_gb300 import inputs as I
from tests.nd_cases import EMPTY, nd_problem

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1601_05725_gb300", "csrc")
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

DRIVER = r"""
#include <cstdio>
#include "solve_internal.h"
size_t bk_gp_smem_limit() { return 160 * 1024; }      // a kernel file's; the plan only compares with it
static std::vector<int32_t> read() {
    int k = 0;
    if (std::scanf("%d", &k) != 1) k = 0;
    std::vector<int32_t> v(k);
    for (auto &x : v) if (std::scanf("%d", &x) != 1) x = 0;
    return v;
}
int main() {
    auto a = read(), colptr = read(), rowind = read(), P = read(), Q = read(), bptr = read(), nd = read();
    bk_plan pl;
    int32_t bad = -1;
    if (bk_plan_build(a[0], colptr.data(), rowind.data(), P.data(), Q.data(), (int32_t)bptr.size() - 1, bptr.data(), a[1],
                      a[2], nd.data(), 1.0, pl, &bad, 0)) return 2;
    bk_solve_plan sp;
    bk_solve_plan_build(pl, sp);
    std::printf("tasks %d %d\n", (int)sp.tasks, pl.n);
    for (auto &T : pl.tasks) std::printf("task %d %d %d %d %d\n", T.lo, T.hi, T.sp_lo, T.level, T.node);
    for (int32_t t : sp.leaf_tasks) std::printf("leaf %d\n", t);
    for (int32_t i : sp.items) std::printf("item %d\n", i);
    std::printf("places %d %d %d\n", sp.tnd0, sp.tf0, sp.tb0);
    for (auto *jobs : {&sp.jobs_a, &sp.jobs_c})
        for (auto &J : *jobs) std::printf("job %d %d %d %d %d\n", J.i0, J.i1, J.lo, J.hi, J.mode);
    for (int32_t i : sp.titems) std::printf("titem %d\n", i);
    return 0;
}
"""


@pytest.fixture(scope="module")
def plan_bin(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None or not os.path.exists(os.path.join(CUDA, "include", "cuda_runtime.h")):
        pytest.skip("no C++ compiler, or no CUDA headers")
    d = tmp_path_factory.mktemp("solve_plan")
    src = d / "drv.cpp"
    src.write_text(DRIVER)
    exe = d / "drv"
    subprocess.run([cxx, "-std=c++17", "-O1", "-w", "-include", "cuda_runtime.h", "-I", os.path.join(CUDA, "include"),
                    "-I", CSRC, str(src), os.path.join(CSRC, "symbolic.cpp"), os.path.join(CSRC, "solve_plan.cpp"),
                    "-o", str(exe)], check=True)
    return str(exe)


def _plan(exe, p):
    nd = p.nd_node_ptr if p.nd_block >= 0 else [0]
    arrs = [[p.n, p.nd_block, p.nd_leaves], p.colptr, p.rowind, p.P, p.Q, p.block_ptr, nd]
    text = "\n".join(f"{len(a)} " + " ".join(str(int(v)) for v in a) for a in arrs)
    out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout
    rec = {}
    for line in out.splitlines():
        k, *v = line.split()
        rec.setdefault(k, []).append([int(x) for x in v])
    return rec


def _check(rec):
    n = rec["tasks"][0][1]
    tasks = rec["task"]
    for lo, hi, sp_lo, level, node in tasks:
        assert (level > 0) == (sp_lo < lo), "a level above the leaves is for separators with rows below them"
    fwd, bwd = np.zeros(n, int), np.zeros(n, int)

    def count(item):
        if item >= 0:
            fwd[item] += item < n
        else:
            bwd[~item] += ~item < n

    for (item,) in rec.get("item", []):
        if -n <= item < n:
            count(item)
    if rec["tasks"][0][0]:
        tnd0, tf0, tb0 = rec["places"][0]
        filled = {}
        for (t,) in rec.get("leaf", []):
            for r in range(tasks[t][0], tasks[t][1]):
                filled[tf0 + r - tnd0] = r
                filled[tb0 + r - tnd0] = ~r
        titems = [v[0] for v in rec.get("titem", [])]
        for i0, i1, lo, hi, mode in rec["job"]:
            for i in range(i0, i1):
                item = titems[i] if mode == 2 else filled.get(i)
                assert item is not None, f"the place of a row of [{lo}, {hi}) is never filled"
                assert lo <= (item if item >= 0 else ~item) < hi
                count(item)
    assert (fwd == 1).all() and (bwd == 1).all()


@pytest.mark.parametrize("name", sorted(EMPTY))
def test_empty_descendants(plan_bin, name):
    sizes, kw = EMPTY[name]
    _check(_plan(plan_bin, nd_problem(5, sizes, **kw)))


@pytest.mark.parametrize("make", [
    lambda: I.netlist_problem(6, n_small=40, m_netlist=600, depth=2),
    lambda: I.netlist_problem(7, n_small=2600, small_sizes=(1, 3), m_netlist=900, depth=3),
    lambda: I.grid_problem(8, k=30, depth=3),
    lambda: I.block_diagonal_problem(9, nblocks=40, size_range=(1, 300)),
    lambda: I.config4(10, n=3000, n_rails=4, rail_deg=(20, 200)),
])
def test_generated_problems(plan_bin, make):
    _check(_plan(plan_bin, make()))
