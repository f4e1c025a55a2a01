"""Small resident rounds inside a thread-block cluster: key spaces at both ends of its range and around them, rounds that stay small,
rounds that grow past what it takes and shrink again, rows walked by four lanes, a warp and the block; against the sorting
route (relations bit for bit, counters equal) and the oracle."""
import numpy as np
import pytest

import oracle
from paper_2609_27203_b200 import synth
from paper_2609_27203_b200 import workloads as W
from tests import helpers as H

pytestmark = pytest.mark.gpu
COUNTERS = ("iterations", "derived_tuples", "candidates", "new_tuples", "improved_tags")


def grid(k):
    at = np.arange(k * k)
    x, y = at % k, at // k
    pairs = [(at[m], at[m] + st) for m, st in ((x > 0, -1), (x < k - 1, 1), (y > 0, -k), (y < k - 1, k))]
    return np.concatenate([a for a, _ in pairs]), np.concatenate([b for _, b in pairs])


def both(prog, out, flags=0, check_oracle=True, **kw):
    from paper_2609_27203_b200 import xlog
    got = []
    for f in (flags, flags | xlog.FLAG_NO_GRAPH, xlog.FLAG_NO_TAG_MIRROR):
        ctx, ids, _ = xlog.load_program(prog, arena_bytes=3 << 30, flags=f | xlog.FLAG_CHECK_INVARIANTS, **kw)
        recs = []
        for _ in range(2):
            recs.append(ctx.fixpoint())
            again = ctx.fixpoint()
            assert again["new_tuples"] == 0 and again["improved_tags"] == 0
            rel = ctx.read(ids[out])
            ctx.reset_idb()
        assert [recs[0][k] for k in COUNTERS] == [recs[1][k] for k in COUNTERS]
        got.append((rel, recs[0]))
        ctx.close()
    for g in got[:2]:
        assert H.compare_relations(g[0], got[2][0], what="cluster vs sorting route")["bit_unequal"] == 0
        assert [g[1][k] for k in COUNTERS] == [got[2][1][k] for k in COUNTERS]
    if check_oracle:
        o, oids, _ = oracle.load_program(prog)
        o.run("seminaive")
        assert H.compare_relations(got[0][0], o.read(oids[out]), what="cluster vs oracle")["bit_unequal"] == 0
    return got[0][1]


@pytest.mark.parametrize("sr", [W.MINPLUS, W.MAXPLUS])
@pytest.mark.parametrize("k,off", [(9, 0), (15, 0), (16, 0), (20, 0), (91, 0), (181, 0), (100, 121071), (100, 121073)])
def test_grids(sr, k, off):                                   # off: node ids up to 2^17 - 1, and past it
    s, d = grid(k)
    w = (1 + 9 * np.random.default_rng(k).random(len(s))).astype(np.float32) * np.float32(1 if sr == W.MINPLUS else -1)
    prog = W.sssp_program(s + off, d + off, w, source=off + k // 2, semiring=sr)
    rec = both(prog, "dist", check_oracle=k < 100)
    assert rec["iterations"] > k


@pytest.mark.parametrize("scale,ef", [(8, 4), (11, 16), (13, 30), (15, 16), (17, 16)])
def test_skewed_graphs_leave_and_come_back(scale, ef):
    s, d, w = synth.rmat_graph(scale, ef, 5 + scale, "u1_10")
    # a long tail behind one node: small rounds after the large ones, longer than the graph is wide
    n = 1 << scale
    tail = np.arange(n - 60, n)
    s, d = np.concatenate([s, tail[:-1]]), np.concatenate([d, tail[1:]])
    w = np.concatenate([w, np.full(59, 0.25, np.float32)])
    key, i = np.unique(s.astype(np.int64) * n + d, return_index=True)
    both(W.sssp_program(s[i], d[i], w[i], source=0), "dist", check_oracle=scale < 15)


@pytest.mark.parametrize("deg", [63, 64, 65, 2047, 2048, 2049, 9000])
def test_fan_out_of_one_row(deg):
    s = np.concatenate([np.zeros(deg, np.int64), 1 + np.arange(deg)])
    d = np.concatenate([1 + np.arange(deg), np.full(deg, deg + 1)])
    w = np.random.default_rng(deg).random(2 * deg).astype(np.float32)
    both(W.sssp_program(s, d, w, source=0), "dist")


def test_many_hubs_in_one_round():                            # more block rows than are queued for the block
    hubs, deg = 600, 2100
    s = np.concatenate([np.zeros(hubs, np.int64), np.repeat(1 + np.arange(hubs), deg)])
    d = np.concatenate([1 + np.arange(hubs), 1000 + (np.repeat(np.arange(hubs), deg) * 7 + np.tile(np.arange(deg), hubs)) % 90000])
    w = np.random.default_rng(1).random(len(s)).astype(np.float32)
    both(W.sssp_program(s, d, w, source=0), "dist", check_oracle=False)


@pytest.mark.parametrize("scale,sources", [(14, 3), (14, 8), (16, 2)])
def test_binary_head_with_a_plain_rule(scale, sources):
    both(W.config5(scale=scale, edge_factor=3, n_sources=sources), "reach", check_oracle=False)


def test_facts_beside_a_rule_without_an_atom_over_the_head_and_the_cap():
    from paper_2609_27203_b200 import xlog
    s, d = grid(60)
    r = np.random.default_rng(2)
    w = (1 + 9 * r.random(len(s))).astype(np.float32)
    prog = W.sssp_program(s, d, w, source=7)
    prog.relations["hint"] = (1, W.MINPLUS)
    prog.rules.insert(0, W.Rule("dist", (W.V(0),), (W.Atom("hint", (W.Var(0),)),)))
    prog.facts["hint"] = ([r.choice(3600, 50, replace=False).astype(np.int32)], (30 * r.random(50)).astype(np.float32))
    prog.facts["dist"] = ([np.arange(0, 3600, 11).astype(np.int32)], (60 * r.random(328)).astype(np.float32))
    rec = both(prog, "dist")
    for cap, ok in ((rec["iterations"], True), (rec["iterations"] - 1, False)):
        ctx, ids, _ = xlog.load_program(prog, arena_bytes=1 << 30, max_iterations=cap)
        if ok:
            ctx.fixpoint()
        else:
            with pytest.raises(xlog.XlogError) as e:
                ctx.fixpoint()
            assert e.value.status == "CONVERGENCE_FAILURE"
        ctx.close()
