"""Patterns whose rows reach little although their band is wide or nothing bounds it: the
traversal's by the sampled reach of their rows; and the same sizes with long searches.  The
route is read from the phase times; results against the oracle."""
import numpy as np
import pytest

import oracle
import synth
from tests.gpu_util import assert_same, oracle_full, to_device

pytestmark = pytest.mark.gpu


def _random(n, per_row, reach, seed, extra=()):
    """Diagonal and per_row entries a row at random distances up to reach on either side."""
    g = np.random.default_rng(seed)
    r = g.integers(0, n, int(per_row * n))
    c = r + g.integers(1, reach + 1, r.size) * g.choice([-1, 1], r.size)
    ok = (c >= 0) & (c < n)
    d = np.arange(n)
    rows, cols = [r[ok], d], [c[ok], d]
    for i in extra:  # rows longer than a search follows
        rows.append(np.full(200, i))
        cols.append(np.clip(i - np.arange(200), 0, n - 1))
    return synth._csr_from_pairs(n, np.concatenate(rows), np.concatenate(cols), "random")


def _chains(n, stride):
    i = np.arange(n)
    a = i[stride:]
    return synth._csr_from_pairs(n, np.concatenate([i, a, a - stride]), np.concatenate([i, a - stride, a]), "chains")


def _traversed(r):
    return r.stats["ms_traverse_global"] > 0


CASES = [
    (lambda: _random(10000, 0.45, 300, 1), True),
    (lambda: _random(30000, 0.9, 700, 2), True),
    (lambda: _random(30000, 1.0, 2000, 3), True),
    (lambda: _chains(20000, 1500), True),
    (lambda: _random(20000, 0.6, 19999, 4), True),             # no band: no search for blocks either
    (lambda: _random(12000, 3.0, 300, 5), False),              # a level wider than a search's queue
    (lambda: _random(9000, 20.0, 600, 6), False),              # eight threads a vertex
    (lambda: _random(30000, 0.45, 300, 7, range(500, 30000, 200)), None),
    (lambda: synth.grid2d(128, 0.8, seed=8), False),
    (lambda: synth.banded(15013, 211, seed=9), False),
    (lambda: synth.grid2d_nd(150, 0.8, seed=10), False),
    (lambda: _random(2048, 0.45, 1500, 11), True),
]


@pytest.mark.parametrize("k", range(len(CASES)))
def test_route_and_result(k):
    import torch
    import paper_2007_00840_gb300 as gs
    make, traversed = CASES[k]
    A = make()
    d = to_device(A)
    r = gs.symbolic_device(*d, opts=gs.options(collect_stats=2))
    if traversed is not None:
        assert _traversed(r) == traversed
    o = oracle_full(A, nthreads=16)
    assert_same(r.to_host(), o)
    out = [torch.empty(A.n, dtype=torch.int32, device="cuda") for _ in range(3)]
    gs.row_counts_noalloc(*d, *out)
    for got, want in zip(out, (np.diff(o["L_rowptr"]), np.diff(o["U_rowptr"]), o["fill_count"])):
        assert np.array_equal(got.cpu().numpy(), want)
    b = gs.batch_device([d, to_device(synth.banded(900, 30, seed=k)), d])
    assert_same(b[0].to_host(), o)
    assert_same(b[2].to_host(), o)


@pytest.mark.parametrize("stride", [400000, 1000])
def test_searches_past_the_bitmap(stride):
    """Orders above the bitmap of a search (1.57 million vertices): rows that reach further back."""
    import paper_2007_00840_gb300 as gs
    d = to_device(_chains(1700000, stride))
    a, b = gs.results_to_host([gs.symbolic_device(*d), gs.symbolic_device(*d, opts=gs.options(frontier_order=2))])
    for k in ("L_rowptr", "L_colidx", "U_rowptr", "U_colidx", "fill_count", "super_start"):
        assert np.array_equal(getattr(a, k), getattr(b, k)), k
