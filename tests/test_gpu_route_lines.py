"""Around the lines between the band, the blocks of a dissection and the traversal: the
orders and entry counts where the route of a call changes, bit-exact against the oracle."""
import numpy as np
import pytest

import oracle
import synth
from tests.gpu_util import assert_same, oracle_full, run_gpu

pytestmark = pytest.mark.gpu


def _near(n, seed):
    """Blocks of about 90 rows with entries near the diagonal, under a last separator that
    reaches everywhere: a band as wide as the matrix and few entries far out."""
    rng = np.random.default_rng(seed)
    top = 12
    i = np.arange(n - top)
    rows = np.repeat(i, 2)
    cols = np.clip(rows + rng.integers(-3, 4, rows.size), rows // 90 * 90, rows // 90 * 90 + 89)
    cols = np.minimum(cols, n - top - 1)
    s = np.repeat(np.arange(n - top, n), 6)
    far = rng.integers(0, n, s.size)
    d = np.arange(n)
    return synth._csr_from_pairs(n, np.concatenate([rows, s, far[::2], d]),
                                 np.concatenate([cols, far, s[::2], d]), "near")


@pytest.mark.parametrize("n", [1599, 1600, 1601, 2599, 2600, 2601, 5003])
def test_dissection_orders(n):
    A = _near(n, n)
    o = oracle_full(A, nthreads=16)
    assert_same(run_gpu(A), o)
    assert_same(run_gpu(A, frontier_order=2), o)


@pytest.mark.parametrize("n,band", [(4095, 700), (4096, 700), (4096, 512), (4096, 511), (7100, 600), (9300, 600)])
def test_wide_bands(n, band):
    A = synth.banded(n, band, seed=n + band)
    o = oracle_full(A, nthreads=16)
    assert_same(run_gpu(A), o)
    assert_same(run_gpu(A, chunk_size=16),
                dict(o, super_start=oracle.supernodes(o["nnzU"], o["L_rowptr"], o["L_colidx"], 16)))
