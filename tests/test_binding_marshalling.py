"""The packed forms of kvd_kv_segment and kvd_store_range arrays have the bytes of the structures (no GPU)."""
import ctypes

import numpy as np
import pytest
import torch

from paper_2603_19664_b200 import binding as B


def _segments(batch, n_segs, segs):
    arr = (B.kvd_kv_segment * (batch * n_segs))()
    for b in range(batch):
        for s, (k, v, stride, first, ln) in enumerate(segs[b]):
            e = arr[b * n_segs + s]
            e.k = k if isinstance(k, int) else None if k is None else k.data_ptr()
            e.v = v if isinstance(v, int) else None if v is None else v.data_ptr()
            e.row_stride, e.first_pos, e.len = int(stride), int(first), int(ln)
    return bytes(arr)


@pytest.mark.parametrize("kind", ["tensors", "addresses", "none", "numpy", "float", "wrapping"])
@pytest.mark.parametrize("batch", [1, 3, 64])
def test_segments(kind, batch):
    t = torch.zeros((4, 64))
    k, v = {"addresses": (1 << 40, 256), "none": (None, None)}.get(kind, (t[1], t[2]))
    num = {"numpy": np.int64, "float": float}.get(kind, int)
    stride = 1 << 33 if kind != "float" else 4096
    first = (1 << 33) + 5 if kind == "wrapping" else 7
    segs = [[(k, v, num(stride), num(first + b), num(b))] * (b % 3) for b in range(batch)]
    n_segs, pos, got = B._marshal_segments(batch, [num(9)] * batch, segs)
    assert n_segs == max(len(s) for s in segs)
    assert bytes(got)[: ctypes.sizeof(B.kvd_kv_segment) * batch * n_segs] == _segments(batch, n_segs, segs)
    assert list(pos) == [9] * batch


@pytest.mark.parametrize("outputs", [True, False])
@pytest.mark.parametrize("n", [0, 1, 64])
def test_ranges(n, outputs):
    t = torch.zeros((4, 64))
    for first in (3, (1 << 32) + 3):
        ranges = [(i, first, 10 + i) + ((t[1], t[2] if i else None) if outputs else ()) for i in range(n)]
        arr = (B.kvd_store_range * max(n, 1))()
        for e, r in zip(arr, ranges):
            e.seq, e.first_row, e.n, e.reserved = r[0], r[1], r[2], 0
            e.k_out, e.v_out = (r[3].data_ptr(), r[4].data_ptr() if r[4] is not None else None) if outputs else (None, None)
        assert bytes(B._marshal_ranges(ranges, outputs))[: 32 * n] == bytes(arr)[: 32 * n]
    if n:
        with pytest.raises(ValueError):
            B._marshal_ranges([(0, 0, 1) if outputs else (0, 0, 1, t, t)], outputs)
