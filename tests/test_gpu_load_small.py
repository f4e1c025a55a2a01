"""Loads at the sizes where one block takes over from the whole device: contents, maxima, order test and rejections.  Exact."""
import numpy as np
import pytest

from paper_2609_27203_b200 import workloads as W

pytestmark = pytest.mark.gpu
SIZES = [1, 2, 31, 33, 1023, 1024, 1025, 8191, 8192, 8193, 300000]


def context():
    from paper_2609_27203_b200 import xlog
    ctx = xlog.Context(arena_bytes=1 << 26)
    return ctx, ctx.relation(2, W.MAXPLUS, "a"), ctx.relation(3, W.LOGSUMEXP, "b")


@pytest.mark.parametrize("n", SIZES)
def test_contents(n):
    ctx, a, b = context()
    rng = np.random.default_rng(n)
    x = np.arange(n, dtype=np.int32) // 3
    cols = [x, np.arange(n, dtype=np.int32) % 3]
    wide = [x, (rng.integers(0, 1 << 24, n)).astype(np.int32), np.arange(n, dtype=np.int32) % 3]      # more than 32 bits together from 86 rows on
    order = np.lexsort(wide[::-1])
    wide = [c[order] for c in wide]
    tags = rng.standard_normal(n).astype(np.float32)
    tags[n // 2] = -0.0
    for rel, c, t in ((a, cols, tags), (a, cols, None), (b, wide, tags)):
        ctx.load(rel, c, t)
        got, gt = ctx.read(rel)
        assert all(np.array_equal(g, w) for g, w in zip(got, c))
        assert np.array_equal(gt, np.zeros(n, np.float32) if t is None else t) and not np.signbit(gt[n // 2])
    ctx.load(a, [c[::-1].copy() for c in cols], tags[::-1].copy())                                   # falling: sorted
    got, gt = ctx.read(a)
    assert all(np.array_equal(g, w) for g, w in zip(got, cols)) and np.array_equal(gt, tags)
    ctx.load(a, [np.concatenate([c, c]) for c in cols], np.concatenate([tags, tags + 1]))            # rising but for one repeat of all
    got, gt = ctx.read(a)
    assert all(np.array_equal(g, w) for g, w in zip(got, cols)) and np.array_equal(gt, tags + 1)
    ctx.close()


@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("at", [0, -1])
def test_one_bad_row_is_found(n, at):
    from paper_2609_27203_b200 import xlog
    ctx, a, _ = context()
    cols = [np.arange(n, dtype=np.int32), np.full(n, 5, np.int32)]
    tags = np.zeros(n, np.float32)
    for what in ("key", "nan", "zero"):
        c, t = [x.copy() for x in cols], tags.copy()
        if what == "key":
            c[1][at] = -1
        else:
            t[at] = np.nan if what == "nan" else -np.inf
        with pytest.raises(xlog.XlogError) as e:
            ctx.load(a, c, t)
        assert e.value.status == "INVALID_VALUE" and ctx.size(a) == 0
    ctx.load(a, cols, tags)                                                                          # and leaves nothing behind
    assert ctx.size(a) == n and np.array_equal(ctx.read(a)[0][0], cols[0])
    if n > 2:                                                                                        # one fall, in the first or the last pair of rows
        c = [x.copy() for x in cols]
        i = 1 if at == 0 else n - 1
        c[0][[i - 1, i]] = c[0][[i, i - 1]]
        t = np.arange(n, dtype=np.float32)
        ctx.load(a, c, t)
        got, gt = ctx.read(a)
        assert np.array_equal(got[0], cols[0]) and gt[i - 1] == i and gt[i] == i - 1
    ctx.close()
