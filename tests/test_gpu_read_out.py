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


@pytest.mark.parametrize("where", ["pinned", "odd address"])
def test_destinations_that_only_a_copy_or_a_mapping_reaches(where):
    """Buffers handed in as device memory that are page-locked host memory (written through its mapping), or that begin between two
    multiples of 4 (copied): as a copy would have it."""
    import torch
    from paper_2609_27203_b200 import xlog
    r = np.random.default_rng(3)
    ctx = xlog.Context(arena_bytes=1 << 24, flags=xlog.FLAG_PROFILE)
    rel = ctx.relation(3, "maxplus")
    ctx.load(rel, [r.integers(0, 1 << 20, 777).astype(np.int32) for _ in range(3)], r.random(777).astype(np.float32))
    hc, ht = ctx.read(rel)
    n = len(ht)
    raw = torch.zeros(4, 4 * n + 16, dtype=torch.uint8, **(dict(pin_memory=True) if where == "pinned" else dict(device="cuda")))
    at = 4 if where == "pinned" else 2
    ptrs = (C.c_void_p * 3)(*[raw[i, at:].data_ptr() for i in range(3)])
    got = C.c_int64()
    torch.cuda.synchronize()
    assert ctx._L.xlog_relation_read(ctx._h, rel, ptrs, raw[3, at:].data_ptr(), n, C.byref(got), xlog.MEM_DEVICE) == 0 and got.value == n
    assert ("k_read_out" in ctx.profile()) == (where == "pinned")
    out = raw.cpu().numpy()
    for i in range(3):
        assert np.array_equal(out[i, at:at + 4 * n].copy().view(np.int32), hc[i])
    assert np.array_equal(out[3, at:at + 4 * n].copy().view(np.float32), ht) and (out[:, :at] == 0).all() and (out[:, at + 4 * n:] == 0).all()
    ctx.close()
