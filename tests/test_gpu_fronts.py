"""Patterns ordered by nested dissection, eliminated block by block on chip (the default
path from 16,384 rows on where the band does not fit).  Bit-exact against the oracle over
several levels, uneven subtrees and one-sided entries, and where the path gives up."""
import numpy as np
import pytest

import oracle
import synth
from tests.gpu_util import assert_same, oracle_full, run_gpu, to_device

pytestmark = pytest.mark.gpu


def _tree(n, leaf, sep, seed, extra=0):
    """Leaves of random sparse blocks under separators of random size whose rows and
    columns reach anywhere in their subtree (not always both ways); a few diagonals missing."""
    rng = np.random.default_rng(seed)
    parts = []

    def add(a, b, lo, hi, k):
        rows = np.repeat(np.arange(a, b), k)
        parts.append((rows, rng.integers(lo, hi, rows.size)))

    def rec(a, b):
        if b - a <= leaf:
            add(a, b, a, b, 3)
            return
        s = int(rng.integers(1, sep))
        m = a + int((b - s - a) * rng.uniform(0.35, 0.65))
        rec(a, m)
        rec(m, b - s)
        add(b - s, b, a, b, 5)
        c, r = parts[-1][0].copy(), rng.integers(a, b, parts[-1][0].size)
        parts.append((r, c))

    rec(0, n)
    if extra:
        parts.append((rng.integers(0, n, extra), rng.integers(0, n, extra)))
    d = np.arange(n)[np.arange(n) % 11 != 0]
    parts.append((d, d))
    return synth._csr_from_pairs(n, np.concatenate([p[0] for p in parts]), np.concatenate([p[1] for p in parts]), "tree")


@pytest.mark.parametrize("n,leaf,sep,extra", [(16384, 60, 12, 0), (20011, 150, 30, 0), (30000, 20, 5, 6), (17000, 400, 3, 0),
                                              (16400, 1500, 40, 0)])
def test_front_trees(n, leaf, sep, extra):
    A = _tree(n, leaf, sep, seed=n + leaf, extra=extra)
    o = oracle_full(A, nthreads=16)
    for chunk in (128, 16):
        ss = o["super_start"] if chunk == 128 else oracle.supernodes(o["nnzU"], o["L_rowptr"], o["L_colidx"], chunk)
        assert_same(run_gpu(A, chunk_size=chunk), dict(o, super_start=ss))


@pytest.mark.parametrize("k,p,leaf", [(129, 0.8, 64), (150, 0.5, 64), (181, 0.9, 16), (230, 0.8, 200)])
def test_front_grids(k, p, leaf):
    A = synth.grid2d_nd(k, p, seed=k, leaf=leaf)
    assert_same(run_gpu(A), oracle_full(A, nthreads=16))


def test_front_gives_up():
    """No closed blocks (one long cycle through a random order), and a vertex above more
    blocks than a row may collect: the traversal's result."""
    rng = np.random.default_rng(1)
    n = 16500
    q = rng.permutation(n)
    A = synth._csr_from_pairs(n, np.concatenate([q, np.arange(n)]), np.concatenate([np.roll(q, 1), np.arange(n)]), "cycle")
    assert_same(run_gpu(A), oracle_full(A, nthreads=16))
    d = np.arange(n)
    i = d[(d % 100 > 0) & (d < n - 1)]
    B = synth._csr_from_pairs(n, np.concatenate([d, i, i - 1, np.full(n, n - 1), d]),
                              np.concatenate([d, i - 1, i, d, np.full(n, n - 1)]), "arrow of blocks")
    assert_same(run_gpu(B), oracle_full(B, nthreads=16))


def test_front_in_batch_and_repeat():
    import paper_2007_00840_gb300 as gs
    mats = [synth.near_square_grid(900, 0.7, seed=2), synth.grid2d_nd(140, 0.8, seed=3), synth.banded(700, 20, seed=4),
            _tree(18000, 100, 20, seed=5)]
    dev = [to_device(A) for A in mats]
    for _ in range(2):
        for A, r in zip(mats, gs.batch_device(dev)):
            assert_same(r.to_host(), oracle_full(A, nthreads=16))
