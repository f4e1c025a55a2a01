"""Candidate tiles at the sizes where their width and who looks their rows up change.  Copies are exact; sums of one fp32 product
per fp64 group against numpy within 1e-6 relative (rounded once to the product, once to the result)."""
import numpy as np
import pytest

from paper_2609_27203_b200 import workloads as W

pytestmark = pytest.mark.gpu
WAVE = 148 * 8 * 256                                          # candidates of one wave of the narrowest tiles


@pytest.mark.parametrize("n", [1, 255, 256, 257, 1025, WAVE - 1, WAVE, WAVE + 1, 3 * WAVE + 77])
def test_one_match_a_row(n):
    from paper_2609_27203_b200 import xlog
    x, y = np.arange(n, dtype=np.int32), (np.arange(n, dtype=np.int64) * 7919 % n).astype(np.int32)
    t = np.random.default_rng(n).standard_normal(n).astype(np.float32)
    prog = W.Program("copy", {"e": (2, W.MAXPLUS), "h": (2, W.MAXPLUS)}, [W.Rule("h", (W.V(1), W.V(0)), (W.Atom("e", (W.Var(0), W.Var(1))),))], {"e": ([x, y], t)}, ("h",))
    ctx, ids, _ = xlog.load_program(prog, arena_bytes=1 << 28, flags=xlog.FLAG_CHECK_INVARIANTS)
    assert ctx.fixpoint()["candidates"] == n
    got, tags = ctx.read(ids["h"])
    order = np.argsort(y, kind="stable")
    assert np.array_equal(got[0], y[order]) and np.array_equal(got[1], x[order]) and np.array_equal(tags, t[order])
    ctx.close()


@pytest.mark.parametrize("n,every,run", [(3, 1, 1), (5000, 1000, 700), (300000, 5, 1), (300000, 5, 6), (2000, 1, 300), (400000, 100000, 200000)])
def test_few_matches_and_long_runs(n, every, run):
    from paper_2609_27203_b200 import xlog
    # h(y, z) :- e(x, y), f(y, z): every `every`-th y has `run` rows of f
    x = np.arange(n, dtype=np.int32)
    ys = np.arange(0, n, every, dtype=np.int32)
    fy, fz = np.repeat(ys, run), np.tile(np.arange(run, dtype=np.int32), len(ys))
    r = np.random.default_rng(run)
    a, b = (0.5 + r.random(n)).astype(np.float32), (0.5 + r.random(len(fy))).astype(np.float32)
    prog = W.Program("join", {"e": (2, W.SUMPROD), "f": (2, W.SUMPROD), "h": (2, W.SUMPROD)},
                     [W.Rule("h", (W.V(1), W.V(2)), (W.Atom("e", (W.Var(0), W.Var(1))), W.Atom("f", (W.Var(1), W.Var(2)))))],
                     {"e": ([x, x], a), "f": ([fy, fz], b)}, ("h",))
    ctx, ids, _ = xlog.load_program(prog, arena_bytes=1 << 29, flags=xlog.FLAG_CHECK_INVARIANTS)
    assert ctx.fixpoint()["candidates"] == len(fy)
    got, tags = ctx.read(ids["h"])
    want = a[fy].astype(np.float64) * b
    assert np.array_equal(got[0], fy) and np.array_equal(got[1], fz) and np.all(np.abs(tags - want) <= 1e-6 * np.abs(want))
    ctx.close()
