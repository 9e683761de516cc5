"""results_to_host copies adjacent arrays as one span only inside one device block: the
blocks of a batch's bands and of its traversed members may be neighbours in memory.  No
GPU: the copies are recorded."""
import types

import pytest

torch = pytest.importorskip("torch")

import paper_2007_00840_gb300 as gs


class _Result:
    """A matrix of order 1 whose six arrays of 64 bytes a field follow those of the results before it."""

    def __init__(self, k, block):
        self.n, self._k, self._b = 1, k, block
        self._owner, self._stream = types.SimpleNamespace(res=None), 0
        self._group, self.stats = "one call", {"traverse_launches": 0}

    def _block(self):
        return self._b

    def _raw(self, name):
        f = gs._FIELDS.index(name)
        wide = name.endswith("rowptr")
        return ((1 << 20) * (f + 1) + 64 * self._k, 8 if wide else 16, "<i8" if wide else "<i4",
                torch.int64 if wide else torch.int32)


@pytest.mark.parametrize("blocks,spans", [([7, 7, 7], 1), ([7, 7, 9], 2), ([7, 9, 7], 3), ([None, None], 2), ([7, None, 7], 3)])
def test_spans_stay_in_their_block(monkeypatch, blocks, spans):
    copied = []

    def as_tensor(cai, device=None):
        i = cai.__cuda_array_interface__
        copied.append((i["data"][0], i["shape"][0], i["typestr"]))
        return torch.zeros(i["shape"][0], dtype=torch.int64 if i["typestr"] == "<i8" else torch.int32)

    empty = torch.empty
    monkeypatch.setattr(torch, "as_tensor", as_tensor)
    monkeypatch.setattr(torch, "empty", lambda n, dtype=None, pin_memory=False: empty(n, dtype=dtype).zero_())
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(synchronize=lambda: None))
    out = gs.results_to_host([_Result(k, b) for k, b in enumerate(blocks)])
    assert len(out) == len(blocks) and len(copied) == 6 * spans
    for ptr, count, typestr in copied:
        first = (ptr % (1 << 20)) // 64
        last = first + count * (8 if typestr == "<i8" else 4) // 64 - 1
        assert len({blocks[k] for k in range(first, last + 1)}) == 1 and (last == first or blocks[first] is not None)
