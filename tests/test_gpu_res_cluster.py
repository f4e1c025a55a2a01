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


def test_many_hubs_in_one_round():                            # long runs in a large relation: grid-wide rounds
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


def profile(prog, **kw):
    from paper_2609_27203_b200 import xlog
    ctx, ids, _ = xlog.load_program(prog, arena_bytes=3 << 30, flags=xlog.FLAG_PROFILE, **kw)
    ctx.fixpoint()
    p = ctx.profile()
    ctx.close()
    return p


def edges(n, deg, seed):
    r = np.random.default_rng(seed)
    key = np.unique(np.repeat(np.arange(n), deg) * n + r.integers(0, n, n * deg))
    s, d = key // n, key % n
    return s, d, (1 + 9 * r.random(len(s))).astype(np.float32)


@pytest.mark.parametrize("sr", [W.MINPLUS, W.MAXPLUS])
@pytest.mark.parametrize("n,deg", [(9000, 3), (60000, 8), (30000, 40), (8000, 64)])
def test_short_runs_leave_with_the_candidates_and_come_back(sr, n, deg):
    """Runs of at most 64: the rounds grow past what a CTA may have, some with few rows and many candidates, and shrink again."""
    s, d, w = edges(n, deg, n)
    w = w if sr == W.MINPLUS else -w
    prog = W.sssp_program(s, d, w, 0, semiring=sr)
    if sr == W.MAXPLUS:                                       # longest paths need a graph without cycles
        keep = s < d
        prog = W.sssp_program(s[keep], d[keep], w[keep], int(s[keep][0]), semiring=sr)
    both(prog, "dist")


def test_a_long_round_is_left_before_it_is_begun():
    # 1, about 64 and about 3,200 rows: the third round has over 190,000 candidates though the second had 4,000
    s, d, w = edges(8000, 64, 3)
    prog = W.sssp_program(s, d, w, 0)
    p, total = profile(prog), both(prog, "dist", check_oracle=False)["candidates"]
    assert "k_res_cluster" in p and p["k_res_expand"]["bytes"] > (total - 50000) * 12


def test_a_first_round_with_many_candidates_is_not_taken():
    # the loaded facts are the first delta: 8,000 rows of 64 matches
    s, d, w = edges(8000, 64, 4)
    prog = W.sssp_program(s, d, w, 0)
    prog.facts["dist"] = ([np.arange(8000, dtype=np.int32)], (np.arange(8000) % 97 + 1).astype(np.float32))
    p = profile(prog)
    assert p["k_res_expand"]["bytes"] > 450000 * 12 and "k_res_count_scan" in p
    both(prog, "dist")


@pytest.mark.parametrize("n,taken", [(16385, True), (16386, False)])
def test_long_runs_only_in_small_relations(n, taken):
    # a star: one run of n - 1 rows, walked by the block
    prog = W.sssp_program(np.zeros(n - 1, np.int32), np.arange(1, n, dtype=np.int32), np.random.default_rng(n).random(n - 1).astype(np.float32) + 1, 0)
    assert ("k_res_cluster" in profile(prog)) == taken
    both(prog, "dist")


@pytest.mark.parametrize("run,taken", [(64, True), (65, False)])
def test_the_longest_run_decides(run, taken):
    s, d, w = edges(20000, 3, run)
    s, d, w = np.append(s, np.zeros(run, int)), np.append(d, 100 + np.arange(run)), np.append(w, np.ones(run, np.float32))
    keep = np.ones(len(s), bool)
    keep[:-run] = s[:-run] != 0                               # node 0 has exactly these
    prog = W.sssp_program(s[keep], d[keep], w[keep], 0)
    assert ("k_res_cluster" in profile(prog)) == taken
    both(prog, "dist", check_oracle=False)


def test_as_many_block_rows_as_a_round_can_have():
    # 7 sources with edges to 4 hubs of 2,300 matches: the second round has 28 rows that the block walks and 64,400 candidates
    hub, leaf = 100 + np.arange(4), 9000 + np.arange(2300)
    s = np.concatenate([np.repeat(np.arange(7), 4), np.repeat(hub, len(leaf))])
    d = np.concatenate([np.tile(hub, 7), np.tile(leaf, 4)])
    w = (1 + np.random.default_rng(1).random(len(s))).astype(np.float32)
    prog = W.reach_program(s.astype(np.int32), d.astype(np.int32), w, np.arange(7, dtype=np.int32))
    p = profile(prog)
    assert "k_res_cluster" in p and p["k_res_expand"]["bytes"] == 0
    both(prog, "reach")
