"""Row-local rounds of sum / logsumexp recursion against the oracle and against the sorting route, counters included.
Sums: the two routes round each round's fp64 sum to fp32 at the same places, so they agree to the rounding of a different
summation order in fp64 (1e-6 relative is over ten fp32 ulps); logsumexp 1e-4 absolute, as everywhere."""
import numpy as np
import pytest

import oracle
from paper_2609_27203_b200 import workloads as W
from tests import helpers as H

pytestmark = pytest.mark.gpu
COUNTERS = ("iterations", "derived_tuples", "candidates", "unique_candidates", "new_tuples", "improved_tags")


def dag(n, m, seed, hub=False):
    r = np.random.default_rng(seed)
    a, b = r.integers(0, n, m), r.integers(0, n, m)
    if hub:                                                   # long runs in both directions: everything into and out of the middle node
        a = np.concatenate([a, np.arange(n // 2), np.full(n - n // 2 - 1, n // 2)])
        b = np.concatenate([b, np.full(n // 2, n // 2), np.arange(n // 2 + 1, n)])
    s, d = np.minimum(a, b), np.maximum(a, b)
    key = np.unique(s.astype(np.int64) * n + d)
    key = key[key // n != key % n]
    return (key // n).astype(np.int32), (key % n).astype(np.int32)


def program(s, d, w, sr, extra):
    p = W.closure_program(s, d, w, sr)
    if extra:                                                 # a second recursive rule over another relation, and loaded facts in the head
        p.relations["f"] = (2, sr)
        p.rules.append(W.Rule("path", (W.V(0), W.V(2)), (W.Atom("path", (W.Var(0), W.Var(1))), W.Atom("f", (W.Var(1), W.Var(2))))))
        p.facts["f"] = ([s[::3].copy(), d[::3].copy()], w[::3].copy())
        p.facts["path"] = ([s[::5].copy(), d[::5].copy()], w[::5].copy())
    return p


@pytest.mark.parametrize("sr", [W.SUMPROD, W.LOGSUMEXP])
@pytest.mark.parametrize("n,m,hub,extra,off", [(2, 4, False, False, 0), (17, 60, False, True, 0), (33, 90, True, False, 0), (300, 700, True, True, 0),
                                               (1025, 2500, False, False, 0), (40, 100, False, False, 8150), (40, 100, True, True, 8152), (40, 100, False, False, 8160)])
def test_rounds_of_one_row(sr, n, m, hub, extra, off):
    from paper_2609_27203_b200 import xlog
    s, d = dag(n, m, n + m, hub)
    s, d = s + np.int32(off), d + np.int32(off)              # values around the largest row that fits (8192)
    w = (0.25 + np.random.default_rng(5).random(len(s))).astype(np.float32)
    if sr == W.SUMPROD and len(w) > 3:
        w[3] = 0.0                                            # the semiring zero: a derivation all the same
    w = w if sr == W.SUMPROD else np.log(w)
    prog = program(s, d, w, sr, extra)
    got = []
    for flags in (0, xlog.FLAG_NO_ROW_FIXPOINT):
        ctx, ids, _ = xlog.load_program(prog, arena_bytes=3 << 30, flags=flags | xlog.FLAG_CHECK_INVARIANTS)
        receipts = [ctx.fixpoint() for _ in range(2)]         # recomputed from the facts, not added
        got.append((ctx.read(ids["path"]), receipts))
        assert receipts[0]["derived_tuples"] == receipts[1]["derived_tuples"]
        ctx.close()
    o, oids, _ = oracle.load_program(prog)
    o.run("seminaive")
    tol = dict(rel_tol=1e-6) if sr == W.SUMPROD else dict(abs_tol=1e-4)
    H.compare_relations(got[0][0], o.read(oids["path"]), what="row sums vs oracle", **tol)
    H.compare_relations(got[0][0], got[1][0], what="row sums vs sorting route", **tol)
    assert [got[0][1][0][k] for k in COUNTERS] == [got[1][1][0][k] for k in COUNTERS]


def test_a_cycle_that_is_long_ends():
    from paper_2609_27203_b200 import xlog
    n = 70
    ctx, ids, _ = xlog.load_program(W.closure_program(np.arange(n), (np.arange(n) + 1) % n, None, W.SUMPROD), arena_bytes=1 << 26)
    with pytest.raises(xlog.XlogError) as e:
        ctx.fixpoint()
    assert e.value.status == "CONVERGENCE_FAILURE"
    ctx.close()
