"""Rules whose groups are products of two runs, against the oracle: forward, receipt and gradient.
Max / min are exact.  Logsumexp 1e-4 absolute, as everywhere.  Sums: fp64 inside a group, one rounding to fp32 per product and
one at the end (1e-6 relative, over ten ulps).  Gradients are fp32 sums of up to a few hundred terms: 1e-4 relative, 1e-5 absolute."""
import numpy as np
import pytest

import oracle
from paper_2609_27203_b200 import workloads as W
from tests import helpers as H

pytestmark = pytest.mark.gpu


def pairs(rng, n, top, fill):
    """Distinct (x, y), x < n, y <= top, about `fill` of all; some x without any."""
    at = rng.random((n, top + 1)) < fill
    at[rng.random(n) < 0.15] = False
    at[0, 0] = at[n - 1, top] = True
    x, y = np.nonzero(at)
    return x.astype(np.int32), y.astype(np.int32)


def program(sr, groups, a_top, b_top, c0, k0, k1, mul, more, seed):
    rng = np.random.default_rng(seed)
    d, e = pairs(rng, groups * mul, a_top, 0.8), pairs(rng, groups * mul + 1, b_top, 0.8)
    tags = lambda n: (0.25 + rng.random(n)).astype(np.float32) if sr == W.SUMPROD else (-4.0 * rng.random(n)).astype(np.float32)
    relations = {"d": (2, sr), "e": (2, sr), "h": (2, sr)}
    terms = (((1, k0),) if k0 else ()) + ((2, k1),)
    rules = [W.Rule("h", (W.Affine(3, ((0, 2),)), W.Affine(c0, terms)), (W.Atom("d", (W.Var(0, mul, 0), W.Var(1))), W.Atom("e", (W.Var(0, mul, 1), W.Var(2)))))]
    facts = {"d": (list(d), tags(len(d[0]))), "e": (list(e), tags(len(e[0])))}
    if more:                                                  # rows of the head that another rule makes, between and inside the groups
        f = pairs(rng, 2 * groups + 5, c0 + k0 * a_top + k1 * b_top, 0.3)
        relations["f"] = (2, sr)
        rules.append(W.Rule("h", (W.V(0), W.V(1)), (W.Atom("f", (W.Var(0), W.Var(1))),)))
        facts["f"] = (list(f), tags(len(f[0])))
    return W.Program("groups", relations, rules, facts, ("h",))


@pytest.mark.parametrize("sr", [W.SUMPROD, W.LOGSUMEXP, W.MAXPLUS, W.MINPLUS])
@pytest.mark.parametrize("groups,a_top,b_top,c0,k0,k1,mul,more", [
    (1, 0, 0, 0, 1, 1, 1, False),                             # one candidate
    (9, 9, 9, 0, 1, 1, 2, False),                             # digit pairs, one block and a group
    (300, 9, 9, 0, 1, 1, 2, True),
    (40, 14, 16, 1, 1, 1, 1, False),                          # 32 slots, runs of up to 17: a whole warp per row
    (40, 15, 15, 0, 1, 1, 3, True),                           # runs of up to 16: half a warp per row
    (33, 80, 31, 0, 0, 1, 1, False),                          # d's column does not reach the head: runs of over 32 rows, the join
    (33, 4, 9, 0, 1, 3, 1, True),                             # slots that only some rows reach
    (33, 10, 11, 10, 1, 1, 1, False),                         # 32 slots with a constant
    (33, 11, 11, 10, 1, 1, 1, False),                         # 33: the sorting route
    (9480, 3, 3, 0, 1, 1, 2, False), (30000, 2, 3, 0, 1, 1, 1, True)])     # one group and more per warp of the whole device
def test_groups(sr, groups, a_top, b_top, c0, k0, k1, mul, more):
    import torch
    from paper_2609_27203_b200 import xlog
    prog = program(sr, groups, a_top, b_top, c0, k0, k1, mul, more, groups + a_top)
    ctx, ids, rules = xlog.load_program(prog, arena_bytes=1 << 28, flags=xlog.FLAG_CHECK_INVARIANTS)
    o, oids, orules = oracle.load_program(prog)
    o.run("seminaive")
    tol = {W.SUMPROD: dict(rel_tol=1e-6), W.LOGSUMEXP: dict(abs_tol=1e-4)}.get(sr, {})
    for _ in range(2):
        receipt = ctx.fixpoint()
        rep = H.compare_relations(ctx.read(ids["h"]), o.read(oids["h"]), what="groups", **tol)
        (d0, _), (e0, _) = prog.facts["d"][0], prog.facts["e"][0]
        nd, ne = (np.bincount(x, minlength=groups * mul + 2) for x in (d0, e0))
        cand = sum(int(nd[p * mul] * ne[p * mul + 1]) for p in range(groups))
        cand += len(prog.facts["f"][1]) if more else 0
        assert receipt["candidates"] == cand and receipt["derived_tuples"] == rep["rows"] and receipt["new_tuples"] == rep["rows"]
    if sr in (W.SUMPROD, W.LOGSUMEXP):
        g = np.random.default_rng(7).standard_normal(rep["rows"]).astype(np.float32)
        parts = ctx.backward(rules[0], torch.from_numpy(g).cuda(), same_buffer_for_same_relation=False)
        for got, want in zip(parts, o.backward(orules[0], g)):
            want = want.astype(np.float64)
            assert np.all(np.abs(got.cpu().numpy() - want) <= 1e-5 + 1e-4 * np.abs(want))
    ctx.close()


def test_a_small_arena_takes_the_sorting_route_or_the_groups_alike():
    from paper_2609_27203_b200 import xlog
    prog = program(W.LOGSUMEXP, 2000, 1, 1, 0, 1, 29, 1, False, 3)          # 31 slots of which four a group are taken
    o, oids, _ = oracle.load_program(prog)
    o.run("seminaive")
    for mb in (4, 64):
        ctx, ids, _ = xlog.load_program(prog, arena_bytes=mb << 20)
        ctx.fixpoint()
        H.compare_relations(ctx.read(ids["h"]), o.read(oids["h"]), abs_tol=1e-4, what="small arena")
        ctx.close()


def whole_values(which, groups, sr, seed):
    """Programs of the same form whose second head column is a sum with negative parts, its value in range for every pair of rows."""
    rng = np.random.default_rng(seed)
    lo, hi, expr = {
        "two dice": (range(1, 7), range(1, 7), (-2, ((1, 1), (2, 1)))),                 # a + b - 2
        "difference": (range(0, 9), range(8, 32), (0, ((1, -1), (2, 1)))),              # b - a
        "twice the difference": (range(3, 7), range(6, 16), (1, ((1, -2), (2, 2)))),
        "by group": (range(0, 3), range(0, 5), (8, ((0, -1), (1, 1), (2, 1)))),         # 8 - p + a + b over p < 9
        "all of them": (range(0, 4), range(5, 9), (10, ((0, -1), (1, -2), (2, 1)))),    # 10 - p - 2 a + b over p < 9
    }[which]
    if which in ("by group", "all of them"):
        groups = min(groups, 9)
    d = np.array([(p, a) for p in range(groups) for a in lo if rng.random() < 0.85 or p == 0], np.int32).T
    e = np.array([(p, b) for p in range(groups) for b in hi if rng.random() < 0.85 or p == 0], np.int32).T
    tags = lambda n: (0.25 + rng.random(n)).astype(np.float32) if sr == W.SUMPROD else (-4.0 * rng.random(n)).astype(np.float32)
    rule = W.Rule("h", (W.V(0), W.Affine(*expr)), (W.Atom("d", (W.Var(0), W.Var(1))), W.Atom("e", (W.Var(0), W.Var(2)))))
    return W.Program("whole values", {k: (2, sr) for k in "deh"}, [rule], {"d": (list(d), tags(d.shape[1])), "e": (list(e), tags(e.shape[1]))}, ("h",))


@pytest.mark.parametrize("sr", [W.SUMPROD, W.LOGSUMEXP, W.MAXPLUS])
@pytest.mark.parametrize("which", ["two dice", "difference", "twice the difference", "by group", "all of them"])
def test_only_the_whole_value_has_to_be_in_range(sr, which):
    import torch
    from paper_2609_27203_b200 import xlog
    prog = whole_values(which, 50, sr, 11)
    ctx, ids, rules = xlog.load_program(prog, arena_bytes=1 << 28, flags=xlog.FLAG_CHECK_INVARIANTS)
    o, oids, orules = oracle.load_program(prog)
    o.run("seminaive")
    ctx.fixpoint()
    tol = {W.SUMPROD: dict(rel_tol=1e-6), W.LOGSUMEXP: dict(abs_tol=1e-4)}.get(sr, {})
    rep = H.compare_relations(ctx.read(ids["h"]), o.read(oids["h"]), what=which, **tol)
    if sr != W.MAXPLUS:
        g = np.random.default_rng(7).standard_normal(rep["rows"]).astype(np.float32)
        parts = ctx.backward(rules[0], torch.from_numpy(g).cuda(), same_buffer_for_same_relation=False)
        for got, want in zip(parts, o.backward(orules[0], g)):
            want = want.astype(np.float64)
            assert np.all(np.abs(got.cpu().numpy() - want) <= 1e-5 + 1e-4 * np.abs(want))
    ctx.close()


@pytest.mark.parametrize("c0,k0", [(-1, 1), (5, -1)])
def test_a_value_out_of_range_is_still_refused(c0, k0):
    from paper_2609_27203_b200 import xlog
    a = np.arange(7, dtype=np.int32)                          # -1 + 0 + 0, and 5 - 6 + 0
    rule = W.Rule("h", (W.V(0), W.Affine(c0, ((1, k0), (2, 1)))), (W.Atom("d", (W.Var(0), W.Var(1))), W.Atom("e", (W.Var(0), W.Var(2)))))
    prog = W.Program("out", {k: (2, W.SUMPROD) for k in "deh"}, [rule], {k: ([0 * a, a], None) for k in "de"}, ("h",))
    ctx, _, _ = xlog.load_program(prog, arena_bytes=1 << 26)
    with pytest.raises(xlog.XlogError) as err:
        ctx.fixpoint()
    assert err.value.status == "CAPACITY_EXCEEDED"
    ctx.close()


@pytest.mark.parametrize("sr", [W.SUMPROD, W.LOGSUMEXP, W.MINPLUS])
@pytest.mark.parametrize("run", [1, 31, 32, 33, 200, 30000])
def test_long_runs_are_spread_over_the_device(sr, run):
    """h(p, b) :- d(p, a), e(p, b): d's column does not reach the head, so nothing but d bounds a group's rows; the group kernels
    take at most 32.  One value in eight of d is missing but the last."""
    import torch
    from paper_2609_27203_b200 import xlog
    r = np.random.default_rng(run)
    there = r.random((3, run)) < 0.875
    there[:, -1] = True
    d, e = [x.astype(np.int32) for x in np.nonzero(there)], [x.astype(np.int32) for x in np.nonzero(np.ones((3, 5)))]
    tags = lambda n: (0.25 + r.random(n)).astype(np.float32) if sr == W.SUMPROD else (-4.0 * r.random(n)).astype(np.float32)
    rule = W.Rule("h", (W.V(0), W.V(2)), (W.Atom("d", (W.Var(0), W.Var(1))), W.Atom("e", (W.Var(0), W.Var(2)))))
    prog = W.Program("runs", {k: (2, sr) for k in "deh"}, [rule], {"d": (d, tags(len(d[0]))), "e": (e, tags(15))}, ("h",))
    ctx, ids, rules = xlog.load_program(prog, arena_bytes=1 << 28, flags=xlog.FLAG_PROFILE)
    o, oids, orules = oracle.load_program(prog)
    o.run("seminaive")
    ctx.fixpoint()
    tol = {W.SUMPROD: dict(rel_tol=1e-6), W.LOGSUMEXP: dict(abs_tol=1e-4)}.get(sr, {})
    rep = H.compare_relations(ctx.read(ids["h"]), o.read(oids["h"]), what=f"runs of {run}", **tol)
    assert rep["rows"] == 15 and ("k_group_rule" in ctx.profile()) == (run <= 32)
    if sr != W.MINPLUS:
        g = r.standard_normal(15).astype(np.float32)
        parts = ctx.backward(rules[0], torch.from_numpy(g).cuda(), same_buffer_for_same_relation=False)
        assert ("k_group_backward" in ctx.profile()) == (run <= 32)
        # against 64 bits: every term is rounded a few times and the sums have up to 26,250 of them, added in fp32 in any order
        want = [np.zeros(len(d[0])), np.zeros(15)]
        head, td, te = ctx.read(ids["h"])[1].astype(np.float64).reshape(3, 5), prog.facts["d"][1].astype(np.float64), prog.facts["e"][1].astype(np.float64).reshape(3, 5)
        size = np.zeros(15)
        for p in range(3):
            at = d[0] == p
            gp = g.reshape(3, 5)[p].astype(np.float64)
            share = np.exp(td[at][:, None] + te[p] - head[p]) if sr == W.LOGSUMEXP else None
            want[0][at] = (share * gp).sum(1) if share is not None else (te[p] * gp).sum()
            want[1].reshape(3, 5)[p] = (share * gp).sum(0) if share is not None else gp * td[at].sum()
            size.reshape(3, 5)[p] = np.abs(share * gp).sum(0) if share is not None else np.abs(gp) * td[at].sum()
        assert np.allclose(parts[0].cpu().numpy(), want[0], rtol=1e-4, atol=1e-5)
        assert np.all(np.abs(parts[1].cpu().numpy() - want[1]) <= 1e-5 + 1e-4 * size)
    ctx.close()
