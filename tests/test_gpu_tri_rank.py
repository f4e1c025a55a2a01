"""Triangle aggregate over the degree-ordered graph against the plain kernels (counts equal; tags to 1e-5 absolute in log space and
1e-6 relative for sums: two roundings of a three-factor fp32 product against two of a three-term fp32 sum of at most 84) and
against closed forms."""
import numpy as np
import pytest

from paper_2609_27203_b200 import synth
from paper_2609_27203_b200 import workloads as W

pytestmark = pytest.mark.gpu


def run(prog, flags=0, arena=1 << 30, again=1):
    from paper_2609_27203_b200 import xlog
    ctx, ids, _ = xlog.load_program(prog, arena_bytes=arena, flags=flags | xlog.FLAG_PROFILE)
    out = []
    for _ in range(again):
        ctx.reset_idb()
        ctx.fixpoint()
        out.append(ctx.read(ids["tri_agg"]))
    ran = "k_tri_rank_small" in ctx.profile()
    ctx.close()
    return out, ran


def sum_program(s, d, w):
    p = W.triangle_program(s, d, w)
    p.relations = {k: (a, W.SUMPROD) for k, (a, _) in p.relations.items()}
    return p


@pytest.mark.parametrize("scale,ef", [(13, 30), (15, 8), (17, 4)])
@pytest.mark.parametrize("sums", [False, True])
def test_against_the_plain_kernels(scale, ef, sums):
    from paper_2609_27203_b200 import xlog
    s, d, w = synth.rmat_graph(scale, ef, scale, "n01")
    assert len(s) >= 1 << 17
    if scale == 13:                                           # the widest tags the products allow
        w[::5] = np.where(w[::5] > 0, 28, -28)
    prog = sum_program(s, d, np.exp(w * 0.1).astype(np.float32)) if sums else W.triangle_program(s, d, w)
    (a, b), ran = run(prog, again=2)
    (want,), plain = run(prog, xlog.FLAG_NO_TRIANGLE_BITMAP)
    assert ran and not plain
    assert all(np.array_equal(x, y) for x, y in zip(a[0], want[0]))
    assert np.allclose(a[1], want[1], rtol=1e-6 if sums else 0, atol=0 if sums else 1e-5)
    assert np.array_equal(a[1].view(np.int32), b[1].view(np.int32))            # run to run, bit for bit


@pytest.mark.parametrize("n", [362, 363, 400, 1025])          # n (n - 1) edges: around 2^17
def test_complete_graph(n):
    s, d = (x.reshape(-1) for x in np.meshgrid(np.arange(n), np.arange(n), indexing="ij"))
    s, d = s[s != d] * 5 + 3, d[s != d] * 5 + 3               # gaps between the ids
    ((got, _), ran) = run(W.triangle_program(s, d, np.zeros(len(s), np.float32)), again=2)
    assert ran == (n * (n - 1) >= 1 << 17)
    cols, tags = got
    assert cols[0].tolist() == (np.arange(n) * 5 + 3).tolist() and (cols[1] == (n - 1) * (n - 2)).all()
    assert np.allclose(tags, np.log((n - 1) * (n - 2)), rtol=1e-6)


def test_hub_wheels_and_lone_nodes():
    # a hub joined both ways to every node of a long directed ring; nodes without in- or out-edges beside it
    from paper_2609_27203_b200 import xlog
    n = 70000
    ring = np.arange(2, n)
    s = np.concatenate([ring, np.zeros(n - 2, int), ring, [0, 1], np.full(500, 1), n + np.arange(300)])
    d = np.concatenate([np.roll(ring, -1), ring, np.full(n - 2, 0), [1, 0], n + 1000 + np.arange(500), np.full(300, 1)])
    w = np.random.default_rng(3).normal(size=len(s)).astype(np.float32)
    prog = W.triangle_program(s, d, w)
    (got,), ran = run(prog)
    (want,), _ = run(prog, xlog.FLAG_NO_TRIANGLE_BITMAP)
    assert ran and all(np.array_equal(x, y) for x, y in zip(got[0], want[0])) and np.allclose(got[1], want[1], rtol=0, atol=1e-5)
    assert got[0][1][0] == n - 2                              # the hub closes one triangle per ring edge


@pytest.mark.parametrize("why", ["loop", "tag", "none"])
def test_graphs_it_leaves_to_the_plain_kernels(why):
    from paper_2609_27203_b200 import xlog
    s, d, w = synth.rmat_graph(13, 30, 9, "n01")
    if why == "loop":
        s, d, w = np.append(s, 5), np.append(d, 5), np.append(w, np.float32(1))
    if why == "tag":
        w[100] = 28.5
    prog = W.triangle_program(s, d, w)
    (got,), ran = run(prog)
    (want,), _ = run(prog, xlog.FLAG_NO_TRIANGLE_BITMAP)
    assert ran == (why == "none")
    assert all(np.array_equal(x, y) for x, y in zip(got[0], want[0])) and np.allclose(got[1], want[1], rtol=0, atol=1e-5)
    if why == "none":                                         # reloading the relation drops the ordered copy
        ctx, ids, _ = xlog.load_program(prog, arena_bytes=1 << 30)
        ctx.fixpoint()
        ctx.load(ids["e"], [s[::2].copy(), d[::2].copy()], w[::2].copy())
        ctx.fixpoint()
        half = ctx.read(ids["tri_agg"])
        (want,), _ = run(W.triangle_program(s[::2], d[::2], w[::2]), xlog.FLAG_NO_TRIANGLE_BITMAP)
        assert all(np.array_equal(x, y) for x, y in zip(half[0], want[0])) and np.allclose(half[1], want[1], rtol=0, atol=1e-5)
        ctx.close()


@pytest.mark.parametrize("why", ["large", "small", "zeros", "edges of the range"])
def test_sums_whose_products_could_leave_the_range(why):
    """Sum-product tags of very different sizes: each corner meets its three factors in another order, and a partial product must not
    overflow or lose bits below the smallest normal number.  The weights have one size per edge class of a tripartite graph, so
    that a whole product is near 1 and every pair of factors is not; against 64 bits."""
    from paper_2609_27203_b200 import xlog
    k, r = 300, np.random.default_rng(4)
    big = {"large": 2.5e19, "small": 6e-20, "zeros": 1e12, "edges of the range": 2.0 ** 41}[why]
    size = [big, big, 1 / big / big] if why in ("large", "small") else [big, 1 / big, 1.0]
    s, d, w = [], [], []
    for part in range(3):                                     # part -> the next part, about half of the pairs
        a, b = np.nonzero(r.random((k, k)) < 0.55)
        s.append(a + part * k)
        d.append(b + (part + 1) % 3 * k)
        w.append((size[part] * r.uniform(0.5, 0.999, len(a))).astype(np.float32))
    s, d, w = np.concatenate(s), np.concatenate(d), np.concatenate(w)
    if why == "zeros":
        w[::7] = 0.0
    assert len(s) >= 1 << 17
    (got,), ran = run(sum_program(s.astype(np.int32), d.astype(np.int32), w))
    assert ran == (why in ("zeros", "edges of the range"))
    m = np.zeros((3 * k, 3 * k))
    there = np.zeros((3 * k, 3 * k))
    m[s, d], there[s, d] = w, 1
    want, cnt = ((m @ m) * m.T).sum(1), ((there @ there) * there.T).sum(1)
    assert np.array_equal(got[0][0], np.arange(3 * k)) and np.array_equal(got[0][1], cnt.astype(np.int32))
    if ran:
        assert np.allclose(got[1], want, rtol=1e-6, atol=0)
    else:                                                     # the plain kernels: the order of an edge list's own corner
        plain, _ = run(sum_program(s.astype(np.int32), d.astype(np.int32), w), xlog.FLAG_NO_TRIANGLE_BITMAP)
        assert np.array_equal(got[1].view(np.int32), plain[0][1].view(np.int32))


def launches(prog, evaluations, reload=False):
    """Kernel names of every evaluation of one context, the graph loaded again before each if `reload`."""
    from paper_2609_27203_b200 import xlog
    ctx, ids, _ = xlog.load_program(prog, arena_bytes=1 << 30, flags=xlog.FLAG_PROFILE)
    out = []
    for _ in range(evaluations):
        if reload:
            ctx.load(ids["e"], *prog.facts["e"])
        ctx.reset_idb()
        ctx.profile_reset()
        ctx.fixpoint()
        out.append((set(ctx.profile()), ctx.read(ids["tri_agg"])))
    ctx.close()
    return out


@pytest.mark.parametrize("why", ["loop", "tag"])
def test_a_graph_that_is_turned_away_pays_for_no_part_of_the_order(why):
    s, d, w = synth.rmat_graph(13, 30, 9, "n01")
    if why == "loop":
        s, d, w = np.append(s, 5).astype(np.int32), np.append(d, 5).astype(np.int32), np.append(w, np.float32(1))
    else:
        w[100] = -28.5
    for ran, _ in launches(W.triangle_program(s, d, w), 3, reload=True):
        assert "k_trk_check" in ran and not ran & {"k_trk_degrees", "k_trk_edges", "k_tri_rank", "k_tri_rank_small"}


@pytest.mark.parametrize("n,m,ordered", [(100000, 140000, False), (4000, 180000, True), (60000, 1000000, True), (250000, 1000000, False), (250000, 1700000, True)])
def test_graphs_on_both_sides_of_the_line(n, m, ordered):
    """Edges spread evenly: few entries to walk, more than 32 an edge, many in all, and many edges; every evaluation of a graph goes
    the same way and gives the same bits."""
    r = np.random.default_rng(n)
    key = np.unique(r.integers(0, n * n, m))
    s, d = (key // n).astype(np.int32), (key % n).astype(np.int32)
    s, d = s[s != d], d[s != d]
    prog = W.triangle_program(s, d, r.standard_normal(len(s)).astype(np.float32))
    got = launches(prog, 3) + launches(prog, 2, reload=True)
    assert ["k_tri_rank_small" in ran for ran, _ in got] == [ordered] * 5
    assert ["k_trk_check" in ran for ran, _ in got] == [True, False, False, True, True]
    for _, (cols, tags) in got[1:]:
        assert all(np.array_equal(x, y) for x, y in zip(cols, got[0][1][0])) and np.array_equal(tags.view(np.int32), got[0][1][1].view(np.int32))


@pytest.mark.parametrize("n", [32767, 32768, 32770, 100003])
@pytest.mark.parametrize("sums", [False, True])
def test_hubs_in_many_units(n, sums):
    """Two hubs joined both ways to the same ring: lists on both sides of the length from which a corner's units are cut finer."""
    from paper_2609_27203_b200 import xlog
    ring = np.arange(2, n + 2)
    pairs = [(ring, np.roll(ring, -1)), (ring[::2], np.roll(ring, 3)[::2])] + [e for h in (0, 1) for e in ((0 * ring + h, ring), (ring, 0 * ring + h))]
    s, d = (np.concatenate([p[i] for p in pairs]).astype(np.int32) for i in (0, 1))
    w = np.random.default_rng(n).normal(size=len(s)).astype(np.float32)
    prog = sum_program(s, d, np.exp(w * 0.1).astype(np.float32)) if sums else W.triangle_program(s, d, w)
    (got, twice), ran = run(prog, again=2)
    (want,), _ = run(prog, xlog.FLAG_NO_TRIANGLE_BITMAP)
    assert ran == (n >= 32768)
    assert all(np.array_equal(x, y) for x, y in zip(got[0], want[0])) and np.allclose(got[1], want[1], rtol=1e-6 if sums else 0, atol=0 if sums else 1e-5)
    assert np.array_equal(got[1].view(np.int32), twice[1].view(np.int32))
