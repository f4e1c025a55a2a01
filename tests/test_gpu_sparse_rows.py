"""Row-local rounds over hash-table rows (short rows, many of them) against the oracle and the sorting route: relations bit for
bit, counters equal.  Row lengths around every table's limit, up to rows that outgrow the last one."""
import numpy as np
import pytest

import oracle
from paper_2609_27203_b200 import workloads as W
from tests import helpers as H

pytestmark = pytest.mark.gpu
COUNTERS = ("iterations", "derived_tuples", "candidates", "new_tuples", "improved_tags")


def forest(n, seed, second=16):
    r = np.random.default_rng(seed)
    child = np.concatenate([np.arange(1, n), r.integers(1, n, n // second)])
    return child, (r.random(len(child)) * child).astype(np.int64)


def chains(lengths):
    """Disjoint paths v -> v+1 -> ...: the first row of a path of k edges holds k tuples."""
    s, at = [], 0
    for k in lengths:
        s += list(range(at, at + k))
        at += k + 1
    s = np.asarray(s)
    return s, s + 1


def graph(name):
    if name == "forest":
        return forest(6000, 3)
    if name == "cycles":                                      # strongly connected pieces of 1 to 40 nodes, tags improve for a while
        r = np.random.default_rng(4)
        s, d, at = [], [], 0
        while at < 4000:
            k = int(r.integers(1, 41))
            s += [at + i for i in range(k)] + [at + int(r.integers(k)) for _ in range(k)]
            d += [at + (i + 1) % k for i in range(k)] + [at + int(r.integers(k)) for _ in range(k)]
            at += k
        return np.asarray(s), np.asarray(d)
    if name == "fans":                                        # runs of r longer than a group of lanes
        r = np.random.default_rng(5)
        hub = np.repeat(np.arange(0, 3000, 100), 90)
        return np.concatenate([np.arange(3000) // 100 * 100 + 1, hub]), np.concatenate([np.arange(3000) // 100 * 100, 10000 + r.integers(0, 5000, len(hub))])
    return chains([int(x) for x in name.split()])


@pytest.mark.parametrize("sr", [W.MAXPLUS, W.MINPLUS])
@pytest.mark.parametrize("name", ["forest", "cycles", "fans", "31 32 33 34 1 2", "127 128 129 255 256 257", "1023 1024", "1025", "1100"])
@pytest.mark.parametrize("spread", [1 << 14, 1 << 16, 1 << 19, 3 << 20])
def test_rows_by_length(sr, name, spread):
    from paper_2609_27203_b200 import xlog
    s, d = graph(name)
    top = int(max(s.max(), d.max())) + 1
    r = np.random.default_rng(len(s))
    ids = np.sort(r.choice(spread, top, replace=False)) if top < spread else np.arange(top)
    if name == "forest":
        r.shuffle(ids)
    ids[ids.argmax()] = spread - 1                            # the largest value of the range
    key = np.unique(ids[s] * spread + ids[d])
    s, d = (key // spread).astype(np.int32), (key % spread).astype(np.int32)
    w = (r.uniform(0.5, 9.5, len(s)) * (-1 if sr == W.MAXPLUS else 1)).astype(np.float32)
    prog = W.closure_program(s, d, w, sr)
    if name == "forest":                                      # facts in the head as well
        prog.facts["path"] = ([s[::7].copy(), d[::7].copy()], (w[::7] * np.float32(0.5)).copy())
    got = []
    for flags in (0, xlog.FLAG_NO_TAG_MIRROR):
        ctx, ids_, _ = xlog.load_program(prog, arena_bytes=9 << 30, flags=flags | xlog.FLAG_CHECK_INVARIANTS)
        rec = ctx.fixpoint()
        assert ctx.fixpoint()["new_tuples"] == 0
        ctx.reset_idb()
        assert ctx.fixpoint()["derived_tuples"] == rec["derived_tuples"]
        got.append((ctx.read(ids_["path"]), rec))
        ctx.close()
    assert H.compare_relations(got[0][0], got[1][0], what="sparse rows vs sorting route")["bit_unequal"] == 0
    assert [got[0][1][k] for k in COUNTERS] == [got[1][1][k] for k in COUNTERS]
    if got[0][1]["unique_candidates"] >= 0:
        assert got[0][1]["unique_candidates"] == got[1][1]["unique_candidates"]
    if spread == 1 << 16:
        o, oids, _ = oracle.load_program(prog)
        o.run("seminaive")
        assert H.compare_relations(got[0][0], o.read(oids["path"]), what="sparse rows vs oracle")["bit_unequal"] == 0


def test_the_iteration_cap_is_reached():
    from paper_2609_27203_b200 import xlog
    s, d = forest(6000, 3)
    for cap in (3, 60):
        ctx, ids, _ = xlog.load_program(W.closure_program((s * 8).astype(np.int32), (d * 8).astype(np.int32), None, W.MINPLUS), arena_bytes=1 << 30, max_iterations=cap)
        if cap == 3:
            with pytest.raises(xlog.XlogError) as e:
                ctx.fixpoint()
            assert e.value.status == "CONVERGENCE_FAILURE"
        else:
            assert ctx.fixpoint()["iterations"] <= cap
        ctx.close()


def descendants(n, seed):
    c, p = forest(n, seed)
    return p, c


def with_fans(n, seed, above):
    """A forest's ancestors, and beside it a node over 50 nodes over 1,200 leaves (three edges to a leaf), under a path of `above`
    nodes that is closed to a ring if it is longer than 1: `above` + 1 rows of over 1,024 tuples."""
    r = np.random.default_rng(seed)
    s, d = forest(n, seed)
    hub, mid, leaf, up = n, n + 1 + np.arange(50), n + 51 + np.arange(1200), n + 1251 + np.arange(above)
    s = np.concatenate([s, 0 * mid + hub, r.choice(mid, 3600), up, up if above > 1 else []]).astype(np.int64)
    d = np.concatenate([d, mid, np.tile(leaf, 3), np.append(up[1:], hub), np.roll(up, -2) if above > 1 else []]).astype(np.int64)
    return s, d


@pytest.mark.parametrize("sr", [W.MAXPLUS, W.MINPLUS])
@pytest.mark.parametrize("name,spread", [("descendants", 1 << 15), ("descendants", 1 << 19), ("one", 1 << 14), ("ring", 1 << 17), ("ring", 1 << 20)])
def test_a_few_long_rows_go_on_alone(sr, name, spread):
    """Rows of over 1,024 tuples beside thousands of short ones: the short ones are finished at once, the long ones round by round,
    with facts in the head as well; relations and counters those of the sorting route."""
    from paper_2609_27203_b200 import xlog
    r = np.random.default_rng(spread)
    s, d = descendants(12000, 5) if name == "descendants" else with_fans(9000, 6, 1 if name == "one" else 7)
    ids = np.sort(r.choice(spread, 12400, replace=False))
    key = np.unique(ids[s] * spread + ids[d])
    s, d = (key // spread).astype(np.int32), (key % spread).astype(np.int32)
    w = (r.uniform(0.5, 9.5, len(s)) * (-1 if sr == W.MAXPLUS else 1)).astype(np.float32)
    prog = W.closure_program(s, d, w, sr)
    prog.facts["path"] = ([s[::5].copy(), d[::5].copy()], (w[::5] * np.float32(0.5)).copy())
    got = []
    for flags in (0, xlog.FLAG_NO_TAG_MIRROR):
        ctx, ids_, _ = xlog.load_program(prog, arena_bytes=9 << 30, flags=flags | xlog.FLAG_CHECK_INVARIANTS | xlog.FLAG_PROFILE)
        rec = ctx.fixpoint()
        assert ("k_sparse_take" in ctx.profile()) == (flags == 0)
        rel = ctx.read(ids_["path"])
        assert ctx.fixpoint()["new_tuples"] == 0
        ctx.reset_idb()
        assert ctx.fixpoint()["derived_tuples"] == rec["derived_tuples"]
        assert H.compare_relations(ctx.read(ids_["path"]), rel)["bit_unequal"] == 0
        got.append((rel, rec))
        ctx.close()
    assert H.compare_relations(got[0][0], got[1][0], what="long rows apart vs sorting route")["bit_unequal"] == 0
    assert [got[0][1][k] for k in COUNTERS + ("unique_candidates",)] == [got[1][1][k] for k in COUNTERS + ("unique_candidates",)]


def test_the_iteration_cap_holds_for_the_long_rows():
    from paper_2609_27203_b200 import xlog
    s, d = with_fans(9000, 6, 40)
    prog = W.closure_program(s.astype(np.int32) * 3, d.astype(np.int32) * 3, None, W.MINPLUS)
    need = None
    for cap in (0, 0, -1, -20):
        ctx, ids, _ = xlog.load_program(prog, arena_bytes=2 << 30, max_iterations=(need or 1000) + cap)
        if cap == 0:
            rec = ctx.fixpoint()
            need = need or rec["iterations"]
            assert rec["iterations"] == need > 21
        else:
            with pytest.raises(xlog.XlogError) as e:
                ctx.fixpoint()
            assert e.value.status == "CONVERGENCE_FAILURE"
        ctx.close()
