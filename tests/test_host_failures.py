"""The library's host code when a call of the runtime or a kernel's status reports a
failure, without a GPU: the library runs over a fake CUDA runtime (fake_cudart.c) in a
process of its own."""
import os
import shutil
import subprocess
import sys

import pytest

from paper_1601_05725_gb300 import build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def fake(tmp_path_factory):
    cc = shutil.which("gcc") or shutil.which("cc")
    if cc is None or shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"):
        pytest.skip("no C or CUDA compiler")
    build.build()
    so = str(tmp_path_factory.mktemp("fake") / "libfake_cudart.so")
    subprocess.run([cc, "-O1", "-shared", "-fPIC", os.path.join(ROOT, "tests", "fake_cudart.c"), "-o", so], check=True)
    return so


def run(fake, body):
    """``body`` in a process over the fake runtime."""
    r = subprocess.run([sys.executable, "-c", "from tests.host_driver import *\n"
                        "from paper_1601_05725_gb300 import inputs as I\n" + body],
                       env=dict(os.environ, LD_PRELOAD=fake, PYTHONPATH=ROOT), cwd=ROOT, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr


PROBLEMS = {
    "grid": "I.grid_problem(3, k=40, depth=2)",
    "netlist": "I.netlist_problem(4, n_small=30, m_netlist=3000, depth=2)",
    "blocks": "I.block_diagonal_problem(5, nblocks=20, size_range=(1, 60))",
}


@pytest.mark.parametrize("name,switch,grown", [
    (name, switch, grown) for name in sorted(PROBLEMS) for switch in (0, 1, 2, 3) for grown in (False, True)
    if not (grown and name == "blocks" and switch % 2)])      # their stored-pattern pass needs no room
def test_wait_that_gave_up_in_a_refactorization(fake, name, switch, grown):
    """No solve with factors that are half new; a refactorization may follow, and starts
    from no stored pattern.  The same when the factors had been given more room."""
    run(fake, f"""
h = Host({PROBLEMS[name]}, refactor_switch={switch})
assert h.factor() == OK and h.solve() == OK and h.refactor() == OK and h.solve() == OK
if {grown}:
    fake.fake_status(0, CAPACITY, 1)
    fake.fake_status(1, GAVE_UP, 1)
else:
    fake.fake_status(0, GAVE_UP, 1)
assert h.refactor() == TIMEOUT
assert h.solve() == NOT_FACTORED
launched()
assert h.refactor() == OK
assert "bk_static_kernel" not in launched()
assert h.solve() == OK and h.refactor() == OK and h.solve() == OK
""")


def test_stages_above_an_empty_level(fake):
    """The stage that goes ahead is launched although no separator of level 1 has rows."""
    run(fake, """
from tests.nd_cases import nd_problem
h = Host(nd_problem(5, [300, 300, 0, 300, 300, 0, 3], chain=True))
launched()
assert h.factor() == OK
assert launched().count("bk_tdesc_kernel") == 2
""")


def test_stored_patterns_serve_again_after_a_jump(fake):
    """A pass that rejects too many pivots turns the stored patterns off until the teams
    alone have moved few."""
    run(fake, """
h = Host(I.grid_problem(3, k=61, depth=2))
assert h.factor() == OK
def stored():
    launched()
    assert h.refactor() == OK
    return "bk_static_kernel" in launched()
assert stored()
fake.fake_status(0, REJECTED, 1000)
assert stored()
fake.fake_status(0, MOVED, 1000)
assert not stored()          # the values jump again
assert not stored()          # the pivots of before hold
assert stored() and stored()
""")


@pytest.mark.parametrize("again", [False, True])
def test_arena_that_outgrows_the_teams(fake, again):
    """Room for the factors that grows past 2^31 entries of L: the complete pass, not the
    teams, whose records hold 31 bits of a place."""
    run(fake, f"""
sizes = np.full(16, 15000)
n = int(sizes.sum())
first = np.isin(np.arange(n), np.cumsum(sizes) - sizes)
r = np.concatenate([np.arange(n), np.flatnonzero(~first)])          # diagonal, and the row below
c = np.concatenate([np.arange(n), np.flatnonzero(~first) - 1])
at = np.lexsort((r, c))
colptr = np.concatenate([[0], np.cumsum(np.bincount(c, minlength=n))])
p = I.Problem("blocks", n, colptr, r[at], np.ones(r.size), np.arange(n), np.arange(n),
              np.concatenate([[0], np.cumsum(sizes)]))
h = Host(p)
assert h.status == OK
call = h.factor
if {again}:
    assert h.factor() == OK
    call = h.refactor
launched()
# every column of L out of room, five times: 10, 104, 480, 1,984, 8,000 entries, then all a block can have
for k in range(5):
    fake.fake_status(k, CAPACITY, 1)
fake.fake_ints(4 * n, 1, 5)
assert call() == OK
seen = launched()
assert seen.count("bk_team_kernel") == 5 and seen.count("bk_gp_task_kernel") == 1, seen
assert h.solve() == OK and h.refactor() == OK and h.solve() == OK
assert "bk_team_kernel" not in launched()
""")


@pytest.mark.parametrize("make", [
    "I.netlist_problem(94, n_small=60, m_netlist=20000, depth=2)",                      # in stages
    "I.netlist_problem(91, n_small=40, m_netlist=6000, depth=1, n_rails=5, rail_deg=(2200, 4000))",   # columns whole
])
def test_no_room_for_the_separator_columns_logs(fake, make):
    """The logs are room a handle can do without: it is made, grows and factors as long as
    the rest fits."""
    run(fake, f"""
import ctypes
p = {make}
def size(h):
    i = basker.Info()
    assert h.L.basker_info(h.h, ctypes.byref(i)) == OK and i.device_bytes == fake.fake_held()
    return i.device_bytes
h = Host(p)
full = size(h)
launched()
assert h.factor() == OK and "bk_tdesc_kernel" in launched()
h.free()
assert fake.fake_held() == 0
def made(cap):
    fake.fake_cap(cap)
    h = Host(p)
    if h.status == OK:
        assert size(h) <= cap and h.factor() == OK
        h.has_logs = "bk_tdesc_kernel" in launched()
    return h
# the least room that a handle is made in (it has no logs), by bisection
lo, hi = 0, full
while hi - lo > 4096:
    mid = (lo + hi) // 2
    h = made(mid)
    lo, hi = (lo, mid) if h.status == OK else (mid, hi)
    h.free()
assert hi < full - 4096, "the handle's own size is the least it is made in"
h = made(hi)
assert not h.has_logs
h.free()
for step in range(1, 8):                 # the logs' own allocations fail, or a later one does
    h = made(hi + (full - hi) * step // 8)
    assert h.status == OK
    h.free()
h = made(full)
assert h.has_logs
# a later call wants room: the logs go
fake.fake_cap(full + 8 * p.n)
assert h.solve() == OK and size(h) < full
launched()
assert h.refactor() == OK and "bk_tdesc_kernel" not in launched()
h.free()
fake.fake_cap(1 << 20)
assert Host(p).status == OOM and fake.fake_held() == 0
""")


@pytest.mark.parametrize("mode", [1, 2])
def test_first_schedule_of_a_handle_without_patterns(fake, mode):
    """A handle from counts alone has no claim order before its first factorization, so
    that one is computed, not checked."""
    run(fake, f"""
n = 8
p = I.Problem("diagonal", n, np.arange(n + 1), np.arange(n), np.ones(n), np.arange(n), np.arange(n), np.array([0, n]))
h = Host(p, symbolic_mode={mode}, factor_mode=1)
launched()
assert h.factor() == OK
seen = launched()
assert "bk_levels_kernel" in seen and "bk_level_check_kernel" not in seen
""")
