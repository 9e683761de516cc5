"""Bands in one batch call and through the server: the edges of words, panels and windows,
with members that have nothing below (or above) the diagonal beside others.  Several
matrices of one call have no stretch cuts, unlike a matrix alone."""
import pytest

import synth

from tests.gpu_util import assert_same, oracle_full, to_device
from tests.test_gpu_band import _edge

pytestmark = pytest.mark.gpu

BANDS = [(0, 0), (0, 40), (40, 0), (1, 1), (0, 31), (0, 33), (33, 64), (0, 700), (0, 1500), (1300, 0), (600, 590), (1400, 1450)]


@pytest.mark.parametrize("n", [1, 31, 32, 33, 64, 65, 129, 517, 1700])
def test_batch_edges(n):
    import paper_2007_00840_gb300 as gs
    mats = [_edge(n, min(bl, n - 1), min(bu, n - 1), seed=n + 10 * k) for k, (bl, bu) in enumerate(BANDS)]
    dev = [to_device(A) for A in mats]
    want = [oracle_full(A) for A in mats]
    for r, o in zip(gs.batch_device(dev), want):
        assert_same(r.to_host(), o)


def test_served_upper_triangles():
    """A burst of patterns without entries below the diagonal, some with them between."""
    import paper_2007_00840_gb300 as gs
    mats = [_edge(200 + 37 * k, 0 if k % 3 else 30, 20 + 11 * k, seed=k) for k in range(24)]
    dev = [to_device(A) for A in mats]
    srv = gs.Server()
    tickets = [srv.submit(*d) for d in dev]
    for t, A in zip(tickets, mats):
        assert_same(srv.wait(t)[0].to_host(), oracle_full(A))
    srv.close()


@pytest.mark.parametrize("cap", [1, 5, 12])
def test_capped_ctas(cap):
    """Under a cap the elimination runs in several launches, or leaves a matrix to the traversal."""
    import paper_2007_00840_gb300 as gs
    opt = gs.options(max_ctas=cap)
    mats = [_edge(900, bl, bu, seed=cap + bl) for bl, bu in [(5, 9), (300, 40), (600, 590), (0, 700), (870, 880)] * 3]
    dev = [to_device(A) for A in mats]
    want = [oracle_full(A) for A in mats]
    for r, o in zip(gs.batch_device(dev, opts=opt), want):
        assert_same(r.to_host(), o)
    for d, o in list(zip(dev, want))[:5]:
        assert_same(gs.symbolic_device(*d, opts=opt).to_host(), o)
    nd = synth.grid2d_nd(130, 0.8, seed=cap)
    assert_same(gs.symbolic_device(*to_device(nd), opts=opt).to_host(), oracle_full(nd, nthreads=16))


def test_bands_and_traversed_members_to_host_together():
    import paper_2007_00840_gb300 as gs
    mats = [A for k in range(6) for A in (_edge(512, 16 * k, 32, seed=k), synth.grid2d_nd(64, 0.8, seed=k))]
    dev = [to_device(A) for A in mats]
    for A, h in zip(mats, gs.results_to_host(gs.batch_device(dev))):
        assert_same(h, oracle_full(A))
