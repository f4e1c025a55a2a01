"""Reading a relation into device tensors: every key width, arity and dictionary column, row counts around the vector width,
destinations at any alignment, columns left out; against the host read of the same relation."""
import ctypes as C

import numpy as np
import pytest

from paper_2609_27203_b200 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("arity,top", [(1, 100), (2, 1 << 15), (2, 1 << 20), (3, 1 << 20), (4, 1 << 16), (2, (1 << 31) - 1)])
@pytest.mark.parametrize("n", [1, 3, 4, 5, 1023, 1025])
def test_device_read_equals_host_read(arity, top, n):
    import torch
    from paper_2609_27203_b200 import xlog
    r = np.random.default_rng(n)
    ctx = xlog.Context(arena_bytes=1 << 24)
    rel = ctx.relation(arity, "maxplus")
    ctx.load(rel, [r.integers(0, top, n).astype(np.int32) for _ in range(arity)], r.random(n).astype(np.float32))
    hc, ht = ctx.read(rel)
    dc, dt = ctx.read_device(rel)
    assert all(np.array_equal(a, b.cpu().numpy()) for a, b in zip(hc, dc)) and np.array_equal(ht, dt.cpu().numpy())
    rows = len(ht)
    buf = torch.full((arity + 1, rows + 8), -7, dtype=torch.int32, device="cuda")
    ptrs = (C.c_void_p * arity)(*[buf[i, 1 + i:].data_ptr() if i != 1 else None for i in range(arity)])     # odd offsets, column 1 left out
    got = C.c_int64()
    assert ctx._L.xlog_relation_read(ctx._h, rel, ptrs, buf[arity, 3:].data_ptr(), rows, C.byref(got), xlog.MEM_DEVICE) == 0 and got.value == rows
    out = buf.cpu().numpy()
    for i in range(arity):
        want = hc[i] if i != 1 else np.full(rows, -7)
        assert np.array_equal(out[i, 1 + i:1 + i + rows], want) and out[i, 1 + i + rows] == -7 and (out[i, :1 + i] == -7).all()
    assert np.array_equal(out[arity, 3:3 + rows].view(np.float32), ht)
    ctx.close()


def test_dictionary_column():
    from paper_2609_27203_b200 import xlog
    p = W.config5(scale=10, n_sources=8)
    ctx, ids, _ = xlog.load_program(p, arena_bytes=1 << 28)
    ctx.fixpoint()
    dc, dt = ctx.read_device(ids["reach"])
    hc, ht = ctx.read(ids["reach"])
    assert all(np.array_equal(a, b.cpu().numpy()) for a, b in zip(hc, dc)) and np.array_equal(ht, dt.cpu().numpy())
    assert set(np.unique(hc[0])) <= set(p.facts["src"][0][0].tolist())
    ctx.close()
