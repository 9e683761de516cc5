"""Tensors of device results hold the result's memory by themselves: after the
result, its siblings of one batch call and the other tensors are gone, and later
calls have reused what was free, their values stand."""
import gc

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2007_00840_gb300 as gs

pytestmark = pytest.mark.gpu

FIELDS = ("L_rowptr", "L_colidx", "U_rowptr", "U_colidx", "fill_count", "super_start")


def _banded(n, b, seed):
    rng = np.random.default_rng(seed)
    rows = [sorted({i} | {int(j) for j in rng.integers(max(0, i - b), min(n, i + b + 1), 3)}) for i in range(n)]
    rp = np.zeros(n + 1, np.int32)
    rp[1:] = np.cumsum([len(r) for r in rows])
    return rp, np.asarray([c for r in rows for c in r], np.int32)


def _cuda(rp, ci):
    return torch.as_tensor(rp, device="cuda"), torch.as_tensor(ci, device="cuda")


@pytest.mark.parametrize("batch", [False, True])
@pytest.mark.parametrize("kept", range(6))
def test_a_tensor_outlives_its_result(batch, kept):
    mats = [_banded(n, 9, n) for n in (1, 33, 400)]
    dev = [_cuda(*m) for m in mats]
    rs = gs.batch_device(dev) if batch else [gs.symbolic_device(*d) for d in dev]
    tensors = [getattr(r, FIELDS[kept]) for r in rs]
    assert all(getattr(r, FIELDS[kept]) is t for r, t in zip(rs, tensors))
    want = [t.cpu().numpy().copy() for t in tensors]
    del rs
    gc.collect()
    last = tensors[2]
    del tensors
    gc.collect()
    for _ in range(3):  # reuse what was given back
        gs.batch_device(dev) if batch else [gs.symbolic_device(*d) for d in dev]
    torch.cuda.synchronize()
    assert last.is_cuda and last.is_contiguous()
    assert last.dtype == (torch.int64 if FIELDS[kept].endswith("rowptr") else torch.int32)
    np.testing.assert_array_equal(last.cpu().numpy(), want[2])


def test_empty_arrays():
    rp = torch.zeros(1, dtype=torch.int32, device="cuda")
    r = gs.symbolic_device(rp, torch.zeros(0, dtype=torch.int32, device="cuda"))
    assert [getattr(r, f).numel() for f in FIELDS] == [1, 0, 1, 0, 0, 1]
    assert r.L_rowptr.cpu().tolist() == [0] and r.L_colidx.dtype == torch.int32
    one = gs.symbolic_device(*_cuda(np.array([0, 1], np.int32), np.array([0], np.int32)))
    assert one.L_colidx.numel() == 0 and one.U_colidx.cpu().tolist() == [0]
