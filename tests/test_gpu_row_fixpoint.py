"""Row-local rounds under max / min at the edges of the rows, against the oracle and the other routes, counters included.  Exact."""
import numpy as np
import pytest

import oracle
from paper_2609_27203_b200 import workloads as W
from tests import helpers as H

pytestmark = pytest.mark.gpu
COUNTERS = ("iterations", "derived_tuples", "candidates", "new_tuples", "improved_tags")


def graph(n, m, seed, hub):
    r = np.random.default_rng(seed)
    s, d = r.integers(0, n, m), r.integers(0, n, m)
    if hub:                                                   # one run far longer than a warp's rows, and one row every round comes back to
        s, d = np.concatenate([s, np.zeros(n, np.int64), np.arange(n)]), np.concatenate([d, np.arange(n), np.zeros(n, np.int64)])
    key = np.unique(s.astype(np.int64) * n + d)
    return (key // n).astype(np.int32), (key % n).astype(np.int32), r.choice(np.float32([0.0, 0.5, 1.0, 2.0, 3.5]), len(key))


@pytest.mark.parametrize("sr", [W.MAXPLUS, W.MINPLUS])
@pytest.mark.parametrize("n,m,hub,off", [(2, 3, False, 0), (31, 60, False, 0), (33, 70, True, 0), (255, 700, False, 0), (257, 500, True, 0), (600, 1800, False, 0),
                                         (40, 90, False, 8150), (40, 90, True, 8152)])
@pytest.mark.parametrize("two", [False, True])
def test_rows(sr, n, m, hub, off, two):
    from paper_2609_27203_b200 import xlog
    s, d, w = graph(n, m, n + m, hub)
    s, d = s + np.int32(off), d + np.int32(off)
    w = -w if sr == W.MAXPLUS else w
    if two:                                                   # two rows a block
        prog = W.odd_even_program(s, d, w, sr)
        outs = ("odd", "even")
    else:
        prog = W.closure_program(s, d, w, sr)
        outs = ("path",)
    o, oids, _ = oracle.load_program(prog)
    o.run("seminaive")
    got = []
    for flags in (0, xlog.FLAG_NO_ROW_FIXPOINT):
        ctx, ids, _ = xlog.load_program(prog, arena_bytes=1 << 30, flags=flags | xlog.FLAG_CHECK_INVARIANTS)
        receipt = ctx.fixpoint()
        for r in outs:
            rep = H.compare_relations(ctx.read(ids[r]), o.read(oids[r]), what=f"{r}, flags {flags}")
            assert rep["bit_unequal"] == 0
        got.append([receipt[k] for k in COUNTERS])
        ctx.close()
    assert got[0] == got[1]
