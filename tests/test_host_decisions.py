"""What the host side decides, without a GPU: api.cu and noalloc.cu compiled as plain C++
over a runtime and launchers that only keep books (host_fake.cpp)."""
import functools
import os
import subprocess

import pytest

from paper_2007_00840_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


@functools.lru_cache(None)
def _program(tmp):
    inc = ["-I", build.INCLUDE, "-I", build.CSRC,
           "-I", os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(build._nvcc()))), "include")]
    src = [os.path.join(build.CSRC, f) for f in ("api.cu", "noalloc.cu")] + [os.path.join(HERE, "host_fake.cpp")]
    exe = os.path.join(tmp, "host_fake")
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-w", "-x", "c++"] + src + inc + ["-o", exe, "-lpthread"])
    return exe


@pytest.fixture(scope="session")
def decide(tmp_path_factory):
    exe = _program(str(tmp_path_factory.mktemp("host")))

    def run(**kw):
        env = dict(os.environ, GSOFA_TIMEOUT_S="0.001") if kw.get("stuck") else None
        out = subprocess.run([exe] + [f"{k}={v}" for k, v in kw.items()], capture_output=True, text=True, timeout=60, env=env)
        assert out.returncode == 0, out.stderr
        return out.stdout.splitlines()
    return run


def _elim(lines):
    """(matrices or parts, CTAs of each, words left, words right) of every band elimination."""
    return [tuple(int(w) for w in (x.split()[1], x.split()[2], x.split()[4], x.split()[6]))
            for x in lines if x.startswith("band_elim")]


@pytest.mark.parametrize("right", [0, 40, 300, 700])
@pytest.mark.parametrize("call", [dict(count=1), dict(count=3), dict(counts=1)])
def test_window_holds_the_next_panel(decide, right, call):
    """A step of the elimination reads the next panel while the panel after the window is
    loaded: the window has to reach one panel down also where no entry is below the diagonal."""
    lines = decide(n=1000, left=0, right=right, **call)
    assert "rc 0" in lines
    assert _elim(lines) and all(left >= 1 for _, _, left, _ in _elim(lines)), lines


def test_unscanned_pattern_is_validated(decide):
    """Where memory runs out before the scan, the traversal checks the rows itself; where the
    scan has checked them, it does not do so again."""
    for at in (0, 1):
        lines = decide(n=1000, left=40, right=40, fail_at=at)
        assert "band_scan" not in lines and "validate" in lines and "rc 0" in lines, (at, lines)
    lines = decide(n=20000, left=15000, right=15000)
    assert "band_scan" in lines and "validate" not in lines and any(x.startswith("trav_class") for x in lines), lines


@pytest.mark.parametrize("below", [2, 1100, 3700])
def test_orders_near_the_largest_index(decide, below):
    """The elimination's loader computes rows of up to LB + 4 panels past the end in 32 bits."""
    n = 2**31 - 1 - below
    assert n + 31 + 32 * (112 + 4) > 2**31 - 1
    assert "band_scan" not in decide(n=n, rows=1, left=3500, right=1)


@pytest.mark.parametrize("cap", [1, 3, 7, 8, 20, 607])
@pytest.mark.parametrize("reach", [30, 300, 700, 1200])
@pytest.mark.parametrize("count", [1, 2, 45])
def test_cap_on_ctas(decide, cap, reach, count):
    """No launch of the elimination has more CTAs than max_ctas; every matrix is eliminated once
    or traversed."""
    lines = decide(n=9000, left=reach, right=reach, count=count, max_ctas=cap, per_row=10)
    assert "rc 0" in lines
    got = _elim(lines)
    assert all(k * c <= cap for k, c, _, _ in got), lines
    if any(x.startswith("trav") for x in lines):
        assert not got and cap < 8 and reach > 30
    else:
        assert got if count == 1 else sum(k for k, _, _, _ in got) == count


@pytest.mark.parametrize("cap", [0, 1, 5, 12, 39, 608])
def test_cap_on_ctas_of_blocks(decide, cap):
    lines = decide(n=20000, left=15000, right=15000, max_ctas=cap, blocks=1)
    got = [tuple(map(int, x.split()[1:3])) for x in lines if x.startswith("front_elim")]
    assert sum(k for k, _ in got) == 40
    if 0 < cap < 608:
        assert all(k * c <= cap for k, c in got), lines
    else:
        assert len(got) == 1


@pytest.mark.parametrize("budget", [1 << 18, 1 << 20, 1 << 22, 1 << 23, 1 << 24, 1 << 25, 0])
def test_budget_of_blocks(decide, budget):
    """The elimination of a dissection holds no more scratch than the traversal's slots might;
    past that the matrix is traversed, with the slots that fit."""
    n = 20000
    lines = decide(n=n, left=15000, right=15000, blocks=1, budget=budget)
    assert "rc 0" in lines and "held 0" in lines
    held = [int(x.split()[4]) for x in lines if x.startswith("front_elim")]
    if budget in (0, 1 << 25):
        assert held
    if held:
        assert budget == 0 or max(held) <= budget // 2 + 5 * n  # besides counters and fill counts
    else:
        assert any(x.startswith("trav_class") for x in lines)


@pytest.mark.parametrize("n,left,reach,traversed", [
    (30000, 1000, 20, True), (30000, 1000, 2000, True), (30000, 1000, 100000, False), (30000, 100, 20, True),
    (30000, 100, 30000, False), (40000, 30, 20, True), (40000, 30, 30000, False), (2047, 1000, 20, True), (900, 300, 20, False)])
def test_route_by_reach(decide, n, left, reach, traversed):
    """A band whose rows reach little is traversed; the same one with long searches is not."""
    lines = decide(n=n, left=left, right=left, reach=reach)
    assert "rc 0" in lines and bool(_elim(lines)) == (not traversed), lines


@pytest.mark.parametrize("n,left,reach,traversed", [
    (30000, 1000, 20, True), (30000, 1000, 1000000, False), (10000, 100, 20, True), (10000, 100, 100000, False),
    (2047, 200, 20, True), (300, 60, 20, False)])
def test_route_of_counts_by_reach(decide, n, left, reach, traversed):
    lines = decide(n=n, left=left, right=left, reach=reach, counts=1)
    assert "rc 0" in lines and bool(_elim(lines)) == (not traversed), lines


def test_no_search_for_blocks_of_short_traversals(decide):
    lines = decide(n=20000, left=15000, right=15000, blocks=1, reach=20)
    assert "front_blocks" not in lines and any(x.startswith("trav_class") for x in lines), lines
    assert "front_blocks" in decide(n=20000, left=15000, right=15000, blocks=1, reach=20000)


@pytest.mark.parametrize("count,traversed", [(2, 2), (5, 5), (20, 0), (120, 0)])
def test_batch_route_by_reach(decide, count, traversed):
    """In a batch only bands that outlast the others are traversed, where the call gains by it."""
    lines = decide(n=30000, left=200, right=200, reach=20, count=count)
    assert "rc 0" in lines and sum(k for k, _, _, _ in _elim(lines)) == count - traversed, lines


@pytest.mark.parametrize("kw", [dict(left=40), dict(left=40, count=5), dict(left=15000, blocks=1), dict(left=15000)])
def test_buffers_of_abandoned_work_are_left_alone(decide, kw):
    """After a wait that ran out, the next call of the thread uses other pinned buffers: the copies
    of the first may still be under way."""
    lines = decide(n=20000, right=kw["left"], stuck=1, **kw)
    assert "first rc -5" in lines and "rc 0" in lines and "in flight" not in lines, lines


@pytest.mark.parametrize("left,per_row,traversed", [(100, 3, True), (100, 4, False), (1500, 4, True)])
def test_bands_of_many_entries_are_searched_where_they_take_long(decide, left, per_row, traversed):
    lines = decide(n=15000, left=left, right=left, reach=20, per_row=per_row)
    assert bool(_elim(lines)) == (not traversed), lines
