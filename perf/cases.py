"""The work the engine is timed on: programs as a user evaluates them through ``paper_2609_27203_b200.xlog``.

A case is a family (``kind``) with its sizes; ``draw`` gives more cases of the same families over the same ranges.  One pass
(``run``) is what a user's program does for one answer or one training step: new facts where each answer comes with new
facts, ``fixpoint``, the derived relation read to device tensors, and for the training step the gradient too.  Sizes are those
of the benchmark's configurations and of the tests' fixtures, or lie between the smallest of the tests and them.

A case stands for one graph up to the numbering of its nodes: the seed numbers the nodes anew, orders rows that come in no
order, and draws every tag.  The derived relations of two seeds thus have as many rows, and no row in common but by chance.
"""
import math

import torch

from paper_2609_27203_b200 import xlog
from paper_2609_27203_b200 import workloads as W

MB, GB = 1 << 20, 1 << 30


def listed():
    return [
        # one training step of the neural-tag program (digit pairs, logsumexp, forward and gradient) at a small batch:
        # all host work, launches and synchronisation
        {"name": "digits_b64", "kind": "digits", "pairs": 64},
        # the same step at the benchmark's batch
        {"name": "digits_b65536", "kind": "digits", "pairs": 65536},
        # all-pairs best path on a small dense-id graph, evaluated afresh (configuration 1)
        {"name": "closure_n1000", "kind": "closure", "nodes": 1000, "edges": 4000},
        # single-source shortest paths, a query with its own source over a resident skewed graph (configuration 2): few, large rounds
        {"name": "sssp_rmat20", "kind": "sssp", "graph": "rmat", "scale": 20, "edge_factor": 16},
        # the same query over a road-like grid: hundreds of small rounds, each waiting for the one before
        {"name": "sssp_grid301", "kind": "sssp", "graph": "grid", "side": 301},
        # reachability from a handful of sources, mid-sized graph
        {"name": "reach_rmat18_s7", "kind": "reach", "scale": 18, "edge_factor": 16, "sources": 7},
        # reachability from 64 sources, the largest configuration (5)
        {"name": "reach_rmat22_s64", "kind": "reach", "scale": 22, "edge_factor": 16, "sources": 64},
        # triangle counts and logsumexp weights per node (configuration 3)
        {"name": "triangles_rmat18", "kind": "triangles", "scale": 18, "edge_factor": 16},
        # materialised triangle join over a hot domain (the worst-case-optimal join's own fixture)
        {"name": "triangle_join_64k", "kind": "triangle_join", "rows": 65536, "domain": 406},
        # materialised four-cycle join, four relations
        {"name": "four_cycle_64k", "kind": "four_cycle", "rows": 65536, "domain": 1024},
        # weighted path sums on an acyclic graph: recursion under logsumexp, tag differences round by round
        {"name": "path_sums_n1000", "kind": "path_sums", "nodes": 1000, "edges": 4000, "semiring": "logsumexp"},
        # new facts every time, unsorted and with repeats, then all ancestors with their best derivation: ids far apart, so
        # the packed keys are wide and nothing is direct-addressed
        {"name": "ancestors_n300k", "kind": "ancestors", "nodes": 300000},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["digits", "closure", "sssp_rmat", "sssp_grid", "reach", "reach_many", "triangles", "triangle_join", "four_cycle",
                       "path_sums", "ancestors"])
    if kind == "digits":
        return {"kind": "digits", "pairs": _log_int(rng, 16, 65536)}
    if kind == "closure":
        n = _log_int(rng, 64, 2500)
        return {"kind": "closure", "nodes": n, "edges": int(n * rng.uniform(1.5, 5.0))}
    if kind == "sssp_rmat":
        return {"kind": "sssp", "graph": "rmat", "scale": rng.randint(12, 20), "edge_factor": rng.randint(4, 16)}
    if kind == "sssp_grid":
        return {"kind": "sssp", "graph": "grid", "side": _log_int(rng, 20, 301)}
    if kind == "reach":
        return {"kind": "reach", "scale": rng.randint(12, 20), "edge_factor": rng.randint(4, 16), "sources": _log_int(rng, 2, 64)}
    if kind == "reach_many":
        return {"kind": "reach", "scale": rng.randint(19, 22), "edge_factor": rng.randint(4, 15), "sources": rng.randint(16, 64)}
    if kind == "triangles":
        return {"kind": "triangles", "scale": rng.randint(10, 18), "edge_factor": rng.randint(4, 15)}
    if kind == "triangle_join":
        rows = _log_int(rng, 1024, 65536)
        return {"kind": "triangle_join", "rows": rows, "domain": max(int(math.sqrt(rows) * math.exp(rng.uniform(math.log(1.6), math.log(30.0)))), 64)}
    if kind == "four_cycle":
        rows = _log_int(rng, 1024, 65536)
        return {"kind": "four_cycle", "rows": rows, "domain": int(math.sqrt(rows) * math.exp(rng.uniform(math.log(4.0), math.log(30.0))))}
    if kind == "path_sums":
        n = _log_int(rng, 64, 1500)
        return {"kind": "path_sums", "nodes": n, "edges": int(n * rng.uniform(1.5, 4.0)), "semiring": rng.choice(["logsumexp", "sumprod"])}
    return {"kind": "ancestors", "nodes": _log_int(rng, 2000, 300000)}


# ---- inputs, made on the device from the seed ---------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _perm(g, n):
    return torch.randperm(n, generator=g, device="cuda")


def _rand(g, n):
    return torch.rand(n, generator=g, device="cuda")


def _i32(x):
    return x.to(torch.int32).contiguous()


def _rmat(base, g, scale, edge_factor, marked=0):
    """Distinct non-loop R-MAT edges (a, b, c, d = .57, .19, .19, .05), ordered by (source, target), and `marked` distinct
    nodes, uniform over all ids but the first, which has edges.  `g` numbers the nodes anew by an exclusive or with one
    number, which keeps neighbouring ids neighbours (R-MAT's hubs sit at neighbouring ids)."""
    n = edge_factor << scale
    src = torch.zeros(n, dtype=torch.int64, device="cuda")
    dst = torch.zeros(n, dtype=torch.int64, device="cuda")
    for _ in range(scale):
        r = _rand(base, n)
        src = (src << 1) | (r >= 0.76)
        dst = (dst << 1) | (((r >= 0.57) & (r < 0.76)) | (r >= 0.95))
    key = torch.unique(((src << scale) | dst)[src != dst])
    nodes = _perm(base, 1 << scale)[:marked]
    if marked:
        nodes[0] = key[torch.randint(key.numel(), (1,), generator=base, device="cuda")] >> scale
    flip = torch.randint(1 << scale, (1,), generator=g, device="cuda")
    key = torch.sort(key ^ ((flip << scale) | flip)).values
    return _i32(key >> scale), _i32(key & ((1 << scale) - 1)), _i32(torch.unique(nodes ^ flip))


def _distinct_pairs(base, g, domain, count, number_a=None, number_b=None):
    """`count` distinct pairs (a, b), a != b, over [0, domain)^2, numbered anew by number_a and number_b (or both by one
    permutation of their own), in no order."""
    space = domain * domain
    if space <= 1 << 22:
        key = _perm(base, space)
    else:
        key = torch.unique(torch.randint(space, (2 * count,), generator=base, device="cuda"))
        key = key[_perm(base, key.numel())]
    key = key[key // domain != key % domain][:count]
    key = key[_perm(g, key.numel())]
    if number_a is None:
        number_a = number_b = _perm(g, domain)
    return _i32(number_a[key // domain]), _i32(number_b[key % domain])


def _log_probs(g, n):
    return math.log(0.5) + (math.log(0.99) - math.log(0.5)) * _rand(g, n)


def _context(program, facts, arena):
    """A context holding the program, its resident facts loaded from device tensors."""
    program.facts = {}
    ctx, ids, rules = xlog.load_program(program, arena_bytes=arena)
    for name, (cols, tags) in facts.items():
        ctx.load(ids[name], cols, tags)
    return ctx, ids, rules


_NONE = [[0], [0], [0.0]]                                    # the program builders want some rows; the facts are loaded apart


def prepare(case, seed):
    base, g = _gen(20609), _gen(seed)
    kind = case["kind"]
    fresh = {}                                               # facts that come anew with every pass
    grad = None
    if kind == "digits":
        b = case["pairs"]
        tags = torch.log_softmax(torch.randn(2 * b, 10, generator=g, device="cuda"), dim=1).reshape(-1).contiguous()
        img = torch.arange(2 * b, dtype=torch.int32, device="cuda").repeat_interleave(10)
        dig = torch.arange(10, dtype=torch.int32, device="cuda").repeat(2 * b)
        program = W.digits_program(torch.zeros(2, 10).numpy())
        ctx, ids, rules = _context(program, {}, 64 * MB + b * 16 * 1024)
        fresh["digit"] = ([img, dig], tags)
        grad = torch.randn(19 * b, generator=g, device="cuda")
        return {"ctx": ctx, "ids": ids, "fresh": fresh, "out": "sum", "rule": rules[0], "grad": grad}
    if kind == "closure":
        n = case["nodes"]
        s, d = _distinct_pairs(base, g, n, case["edges"])
        ctx, ids, _ = _context(W.closure_program(*_NONE), {"edge": ([s, d], _log_probs(g, s.numel()))}, 256 * MB + n * n * 128)
        return {"ctx": ctx, "ids": ids, "fresh": fresh, "out": "path"}
    if kind == "sssp":
        if case["graph"] == "rmat":
            s, d, source = _rmat(base, g, case["scale"], case["edge_factor"], 1)
        else:                                                # four neighbours, both directions
            k = case["side"]
            at = torch.arange(k * k, device="cuda")
            x, y = at % k, at // k
            pairs = [(at[m], at[m] + step) for m, step in ((x > 0, -1), (x < k - 1, 1), (y > 0, -k), (y < k - 1, k))]
            s, d = torch.cat([a for a, _ in pairs]), torch.cat([b for _, b in pairs])
            o = torch.argsort(s * (k * k) + d)
            s, d = _i32(s[o]), _i32(d[o])
            source = torch.randint(k * k, (1,), generator=g, device="cuda", dtype=torch.int32)
        w = 1.0 + 9.0 * _rand(g, s.numel())
        ctx, ids, _ = _context(W.sssp_program(*_NONE), {"edge": ([s, d], w)}, 512 * MB + s.numel() * 128)
        fresh["dist"] = ([source], torch.zeros(1, device="cuda"))
        return {"ctx": ctx, "ids": ids, "fresh": fresh, "out": "dist"}
    if kind == "reach":
        s, d, srcs = _rmat(base, g, case["scale"], case["edge_factor"], case["sources"])
        w = 1.0 + 9.0 * _rand(g, s.numel())
        carried = 1 << (max(case["sources"] - 1, 1)).bit_length()
        ctx, ids, _ = _context(W.reach_program(*_NONE, [0]), {"edge": ([s, d], w)},
                               768 * MB + s.numel() * 72 + (carried << case["scale"]) * 36)
        fresh["src"] = ([srcs], None)
        return {"ctx": ctx, "ids": ids, "fresh": fresh, "out": "reach"}
    if kind == "triangles":
        s, d, _ = _rmat(base, g, case["scale"], case["edge_factor"])
        ctx, ids, _ = _context(W.triangle_program(*_NONE), {"e": ([s, d], torch.randn(s.numel(), generator=g, device="cuda"))},
                               256 * MB + s.numel() * 256)
        return {"ctx": ctx, "ids": ids, "fresh": fresh, "out": "tri_agg"}
    if kind in ("triangle_join", "four_cycle"):
        names = ["r", "s", "t"] if kind == "triangle_join" else ["r", "s", "t", "u"]
        facts = {}
        number = [_perm(g, case["domain"]) for _ in names]   # one numbering for the values of each variable
        for i, name in enumerate(names):
            a, b = _distinct_pairs(base, g, case["domain"], case["rows"], number[i], number[(i + 1) % len(names)])
            facts[name] = ([a, b], _log_probs(g, a.numel()))
        build = W.triangle_join_program if kind == "triangle_join" else W.four_cycle_program
        rows, dom = case["rows"], case["domain"]
        out = rows ** len(names) / dom ** len(names)
        ctx, ids, _ = _context(build(*([_NONE] * len(names))), facts, int(512 * MB + 64 * out + 128 * rows * rows / dom))
        return {"ctx": ctx, "ids": ids, "fresh": fresh, "out": "tri" if kind == "triangle_join" else "c4"}
    if kind == "path_sums":
        n = case["nodes"]
        a, b = _distinct_pairs(base, base, n, case["edges"])
        key = torch.unique(torch.minimum(a, b).long() * n + torch.maximum(a, b))    # every edge one way: no cycle
        number, w = _perm(g, n), 0.25 + _rand(g, key.numel())
        sr = case["semiring"]
        ctx, ids, _ = _context(W.closure_program(*_NONE, semiring=sr), {"edge": ([_i32(number[key // n]), _i32(number[key % n])], w.log() if sr == "logsumexp" else w)},
                               256 * MB + n * n * 128)
        return {"ctx": ctx, "ids": ids, "fresh": fresh, "out": "path"}
    # ancestors: every node but the first has a parent among the nodes before it, one in sixteen a second one; node numbers
    # shuffled; a quarter of the rows said twice; no order
    n = case["nodes"]
    child = torch.cat([torch.arange(1, n, device="cuda"), torch.randint(1, n, (n // 16,), generator=base, device="cuda")])
    parent = (_rand(base, child.numel()).double() * child).long()
    child, parent = torch.cat([child, child[: n // 4]]), torch.cat([parent, parent[: n // 4]])
    name, o = _perm(g, n), _perm(g, child.numel())
    ctx, ids, _ = _context(W.closure_program(*_NONE, name="ancestors"), {}, 4 * GB)
    fresh["edge"] = ([_i32(name[child[o]]), _i32(name[parent[o]])], _log_probs(g, child.numel()))
    return {"ctx": ctx, "ids": ids, "fresh": fresh, "out": "path"}


def run(state):
    ctx, ids = state["ctx"], state["ids"]
    if state["fresh"]:
        for name, (cols, tags) in state["fresh"].items():
            ctx.load(ids[name], cols, tags)                  # drops what was derived before
    else:
        ctx.reset_idb()
    ctx.fixpoint()
    out = ctx.read_device(ids[state["out"]])
    if "grad" in state:
        return out, ctx.backward(state["rule"], state["grad"])[0]
    return out


def work(case):
    """Bytes: every input row once (4 per column and tag), every row of the result once.  Flops: one otimes and one oplus per
    derivation.  Sizes of results are the expected ones."""
    kind = case["kind"]
    if kind == "digits":
        b = case["pairs"]
        return {"bytes": b * (20 * 12 + 19 * 12 + 19 * 4 + 20 * 4), "flops": 4 * 100 * b}
    if kind == "closure":
        n, m = case["nodes"], case["edges"]
        return {"bytes": m * 12 + 0.9 * n * n * 12, "flops": 2 * 0.9 * n * m}
    if kind == "sssp":
        n = 1 << case["scale"] if case["graph"] == "rmat" else case["side"] ** 2
        m = case["edge_factor"] * n if case["graph"] == "rmat" else 4 * n
        return {"bytes": m * 12 + 0.5 * n * 8, "flops": 2 * m}
    if kind == "reach":
        n = 1 << case["scale"]
        m, rows = case["edge_factor"] * n, 0.25 * n * case["sources"]
        return {"bytes": m * 12 + rows * 12, "flops": 2 * rows * 2 * case["edge_factor"]}
    if kind == "triangles":
        n = 1 << case["scale"]
        m = case["edge_factor"] * n
        return {"bytes": m * 12 + 0.33 * n * 12, "flops": 3 * 4.0 * m * case["edge_factor"] / 2}
    if kind in ("triangle_join", "four_cycle"):
        k = 3 if kind == "triangle_join" else 4
        rows = (case["rows"] / case["domain"]) ** k
        return {"bytes": k * case["rows"] * 12 + rows * (k + 1) * 4, "flops": (k - 1) * rows}
    if kind == "path_sums":
        n, m = case["nodes"], case["edges"]
        return {"bytes": m * 12 + 0.1 * n * n * 12, "flops": 2 * 0.1 * n * m}
    n = case["nodes"]
    return {"bytes": 1.3 * n * 12 + 20 * n * 12, "flops": 2 * 20 * n}


def tolerance(case):
    # max-plus and min-plus over linear rules have one fp32 fixpoint, and the joins one product per row: bit for bit.
    # logsumexp and sums against the same in 64 bits: 4e-8 to 1.4e-7 off (the gradients most), single values up to 1.2e-6
    if case["kind"] in ("digits", "triangles", "path_sums"):
        return {"rel": 6e-7, "max": 1e-5}
    return "exact"
