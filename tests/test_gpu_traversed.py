"""The traversal's own paths on patterns that nothing eliminates: unstructured ones, whose
rows reach little.  (Grids, bands and dissections of the other tests are eliminated by default, so
that the batch autotuner, the counts call near its largest order, and a server's space
budget and host logs are reached through these.)  And a dissection inside a batch that is
large enough to be eliminated there."""
import numpy as np
import pytest

import oracle
import synth
from tests.gpu_util import assert_same, oracle_full, oracle_full_cached, to_device
from tests.test_gpu_reach import _random

pytestmark = pytest.mark.gpu

FIELDS = ("L_rowptr", "L_colidx", "U_rowptr", "U_colidx", "fill_count", "super_start")


def _far(n, per_row, seed, dense=()):
    """Unstructured; dense: rows with an entry in every second column."""
    A = _random(n, per_row, n - 1, seed)
    if not len(dense):
        return A
    r = np.repeat(np.arange(n), np.diff(A.rowptr))
    rows, cols = [r], [A.colidx.astype(np.int64)]
    for i in dense:
        cols.append(np.arange(0, n, 2))
        rows.append(np.full(cols[-1].size, i))
    return synth._csr_from_pairs(n, np.concatenate(rows), np.concatenate(cols), "far")


def test_counts_with_fewer_ctas():
    """The largest order: the overflow lists of a full grid do not fit the fixed scratch; the last
    row's first level of 32,767 vertices is longer than the list on chip."""
    import torch
    import paper_2007_00840_gb300 as gs
    from paper_2007_00840_gb300._lib import GSOFA_NOALLOC_MAX_N as n
    A = _far(n, 0.5, 21, dense=[n - 1])
    o = oracle.symbolic(A, nthreads=16)
    want = (o["nnzL"], o["nnzU"], oracle.fill_count(A, o["nnzL"], o["nnzU"]))
    d = to_device(A)
    for _ in range(2):
        out = [torch.zeros(n, dtype=torch.int32, device="cuda") for _ in range(3)]
        gs.row_counts_noalloc(*d, *out)
        for g, w in zip(out, want):
            assert np.array_equal(g.cpu().numpy(), np.asarray(w, np.int32))


def test_autotuned_batch():
    import paper_2007_00840_gb300 as gs
    mats = [_far(int(n), 0.7, k) for k, n in enumerate(np.linspace(2600, 6000, 12))]
    mats += [synth.grid2d_nd(k, 0.8, seed=k) for k in (60, 75, 90)]
    dev = [to_device(A) for A in mats]
    for _ in range(2):  # tuned, then replayed
        res = gs.batch_device(dev, opts=gs.options(autotune=1))
        for A, h in zip(mats, gs.results_to_host(res)):
            assert_same(h, oracle_full(A))


def test_dissection_in_a_batch():
    import paper_2007_00840_gb300 as gs
    mats = [synth.grid2d(40, 0.7, seed=1), synth.grid2d_nd(262, 0.8, seed=2), _far(70000, 0.6, 3)]
    res = gs.batch_device([to_device(A) for A in mats], opts=gs.options(collect_stats=2))
    assert res[1].stats["ms_traverse"] > 0 and res[1].stats["ms_traverse_global"] == 0  # eliminated
    assert res[2].stats["ms_traverse_global"] > 0
    for k, (A, r) in enumerate(zip(mats, res)):
        assert_same(r.to_host(), oracle_full_cached(("traversed", k), A))


@pytest.mark.parametrize("mode", ["fewer slots", "host logs"])
def test_served_space_budget(mode):
    """A large unstructured request under a cap that leaves it few class slots, or none whole."""
    import paper_2007_00840_gb300 as gs
    n = 90000
    big = _far(n, 0.8, 5)
    small = [synth.batch_mix_one(m, seed=50 + m, n_lo=200, n_hi=2000) for m in range(4)]
    dev = [to_device(A) for A in [big] + small]
    base = 96 * n + 8 * (64 * big.nnz + 16 * n) + (1 << 20)  # its charge without slots
    slot = (n + 1023) // 1024 * 1024
    cap = base + (40 * (slot // 8 + slot // 256 + 4 * slot) if mode == "fewer slots" else 8 * (slot // 8 + slot // 256))
    srv = gs.Server(mem_cap_bytes=cap, streams=1)
    tickets = [srv.submit(*d) for d in dev]
    for k, (t, A) in enumerate(zip(tickets, [big] + small)):
        assert_same(srv.wait(t)[0].to_host(), oracle_full_cached(("served budget", k), A))
    st = srv.stats()
    assert st["completed"] == len(dev) and st["failed"] == 0
    assert st["peak_mem_in_use"] <= cap and 0 < st["peak_device_bytes"] <= cap
    srv.close()
