"""Banded matrices by elimination in shared memory: the default path wherever the band
fits on chip.  Bit-exact against the oracle at the edges of its words (32 columns), panels
(32 rows), clusters and supernode groups, and beside matrices that do not fit."""
import numpy as np
import pytest

import oracle
import synth
from tests.gpu_util import assert_same, oracle_full, run_gpu, to_device

pytestmark = pytest.mark.gpu


def _pairs(n, rows):
    p = np.array([(i, j) for i in range(n) for j in rows(i) if 0 <= j < n], dtype=np.int64).reshape(-1, 2)
    return synth._csr_from_pairs(n, p[:, 0], p[:, 1], "band")


def _edge(n, bl, bu, seed):
    """Rows that reach exactly bl left and bu right somewhere, with a few entries between."""
    rng = np.random.default_rng(seed)
    def rows(i):
        a = rng.integers(i - bl, i + bu + 1, 3).tolist()
        return a + ([i] if i % 5 else []) + ([i - bl] if i % 3 == 0 else []) + ([i + bu] if i % 4 == 0 else [])
    return _pairs(n, rows)


@pytest.mark.parametrize("bl,bu", [(0, 0), (0, 40), (40, 0), (1, 1), (31, 32), (32, 31), (33, 64), (95, 97)])
def test_band_word_edges(bl, bu):
    for n in (1, 2, 31, 32, 33, 63, 64, 65, 127, 128, 129, 517):
        A = _edge(n, min(bl, n - 1), min(bu, n - 1), seed=n + 1000 * bl + bu)
        assert_same(run_gpu(A), oracle_full(A))


@pytest.mark.parametrize("b", [255, 256, 257, 300, 511, 512, 513, 600, 1100, 1500])
def test_band_cluster_sizes(b):
    """One CTA up to 8 words of band, then clusters of 4 and 8."""
    A = _edge(1700, b, max(1, b - 40), seed=b)
    o = oracle_full(A)
    assert_same(run_gpu(A), o)
    B = _edge(1700, max(1, b // 7), b, seed=b + 1)
    assert_same(run_gpu(B), oracle_full(B))


def test_band_shapes():
    rng = np.random.default_rng(3)
    cases = [
        _pairs(3000, lambda i: [i] + ((i // 48) * 48 + rng.integers(0, 48, 3)).tolist()),             # blocks: many stretches
        _pairs(3000, lambda i: [i] + ((i // 64) * 64 + rng.integers(0, 64, 3)).tolist() + [i + 90]),  # blocks, entries right of them
        _pairs(900, lambda i: [i, i + 1, i + 7]),                                                      # nothing below the diagonal
        _pairs(900, lambda i: [i, i - 1, i - 40]),                                                     # nothing above it
        _pairs(400, lambda i: []),                                                                     # no entries
        _pairs(160, lambda i: range(160)),                                                             # more entries than are staged
        _pairs(900, lambda i: range(i - 70, i + 71, 3) if i % 97 == 0 else [i - 33, i + 64]),
    ]
    for A in cases:
        o = oracle_full(A)
        for chunk in (128, 1, 48, 1024):
            h = run_gpu(A, chunk_size=chunk)
            ss = o["super_start"] if chunk == 128 else oracle.supernodes(o["nnzU"], o["L_rowptr"], o["L_colidx"], chunk)
            assert_same(h, dict(o, super_start=ss)), (A.n, chunk)


def test_band_batch_mixed():
    """A batch of one-CTA bands, clusters and matrices whose band does not fit, results in order."""
    import paper_2007_00840_gb300 as gs
    mats = [_edge(700, 30, 30, 1), synth.random_pattern(2500, 0.002, seed=4), _edge(900, 600, 590, 2), _edge(33, 5, 3, 3),
            synth.grid2d_nd(110, 0.8, seed=5), _edge(1500, 1400, 1450, 6), synth.near_square_grid(2000, 0.7, seed=7),
            _edge(1, 0, 0, 8)]
    dev = [to_device(A) for A in mats]
    for opt in (None, gs.options(chunk_size=16)):
        for A, r in zip(mats, gs.batch_device(dev, opts=opt)):
            o = oracle_full(A)
            ss = o["super_start"] if opt is None else oracle.supernodes(o["nnzU"], o["L_rowptr"], o["L_colidx"], 16)
            assert_same(r.to_host(), dict(o, super_start=ss))


def test_band_and_traversal_agree():
    """The same call with a traversal option set runs the traversal: same bytes."""
    for A in (_edge(2000, 70, 90, 9), synth.banded(4000, 150, seed=2), synth.grid2d(50, 0.6, seed=4)):
        a, b = run_gpu(A), run_gpu(A, frontier_order=2)
        for k in ("L_rowptr", "L_colidx", "U_rowptr", "U_colidx", "fill_count", "super_start"):
            assert np.array_equal(getattr(a, k), getattr(b, k)), k
