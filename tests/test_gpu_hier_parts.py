"""The hierarchical variant at the largest parts, whose local searches fill their maps, against
the oracle."""
import numpy as np
import pytest

from paper_1607_07696_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def rn():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1607_07696_gb300 import rn as RN

    return RN


def same(got, ref):
    return len(got[0]) == len(ref) and all(
        np.array_equal(x, y.astype(x.dtype)) for x, y in zip(got, (ref.u, ref.v, ref.d)))


def lattice(wd, ht, seed):
    """A full lattice (at most four arcs a node) with weights around 100."""
    e = I.full_grid(wd, ht, 1)
    e.w = np.random.default_rng(seed).integers(60, 141, size=e.m).astype(np.uint32)
    return e


@pytest.mark.parametrize("wd,ht,part", [(99, 165, 4096), (115, 220, 6400), (127, 205, 6516)])
def test_parts_searched_whole(rn, oracle, wd, ht, part):
    """Nodes without overflow rows, parts that start inside a page, a bound that covers the part:
    four warps insert every page of a part into its map, and a slot that one of them drew in
    vain is out of use while the last page is inserted."""
    e = lattice(wd, ht, wd)
    g = rn.rn_graph_load(e.src, e.dst, e.w, e.n)
    og = oracle.graph(e.n, e.src, e.dst, e.w)
    R, S = I.disjoint_sets(e.n, 3000, 12, ht)
    ref = og.join(S, R, rn.RN_THETA_MAX)  # (from the few: d(u, v) = d(v, u))
    o = np.lexsort((ref.u, ref.v))
    for run in range(3):
        u, v, d = rn.rn_distance_join_hier(g, R, S, rn.RN_INF, part)
        assert 3000 < rn.rn_last_hier_stats()["max_part"] <= part
        assert np.array_equal(u, ref.v[o]) and np.array_equal(v, ref.u[o]) and np.array_equal(d, ref.d[o].astype(d.dtype)), run


def caves(n, size, hub, seed):
    """Groups of `size` nodes, each joined to all of its group (so that its arcs stay near it in
    any order by neighbourhoods), consecutive groups joined by two edges, and one node of `hub` arcs."""
    e = set()
    for b in range(0, n, size):
        top = min(b + size, n)
        e |= {(i, j) for i in range(b, top) for j in range(i + 1, top)}
        e |= {(top - 1, top), (top - 2, top + 1)} if top + 1 < n else set()
    mid = n // 2 // size * size
    e |= {(mid, mid + size + i) for i in range(hub - size + 1)}
    e = np.array(sorted(e), np.int64)
    w = np.random.default_rng(seed).integers(1, 1000, size=len(e))
    return I.EdgeList(n, e[:, 0].astype(np.uint32), e[:, 1].astype(np.uint32), w.astype(np.uint32), None, {})


@pytest.mark.parametrize("size,hub,part", [
    (20, 24, 6500),  # two overflow rows a node: a part's pages fit
    (41, 60, 6500),  # five, and eight for one node: eight for each do not fit
    (41, 60, 2048),  # in smaller parts they do
])
def test_parts_of_overflow_rows(rn, oracle, size, hub, part):
    a, b = caves(11_000, size, hub, size), lattice(400, 475, size)  # (most nodes need no overflow row)
    e = I.EdgeList(a.n + b.n, np.r_[a.src, b.src + a.n, 0].astype(np.uint32), np.r_[a.dst, b.dst + a.n, a.n].astype(np.uint32),
                   np.r_[a.w, b.w, 5].astype(np.uint32), None, {})
    g = rn.rn_graph_load(e.src, e.dst, e.w, e.n)
    og = oracle.graph(e.n, e.src, e.dst, e.w)
    rng = np.random.default_rng(hub)
    pick = np.r_[rng.permutation(a.n)[:300], a.n + rng.permutation(b.n)[:1500]]
    pick = rng.permutation(pick)
    R, S = pick[:700], pick[700:]
    for theta in (800, 4_000):
        ref = og.join(R, S, theta)
        assert len(ref) > 100
        assert same(rn.rn_distance_join_hier(g, R, S, theta, part), ref), theta
        assert part / 2 < rn.rn_last_hier_stats()["max_part"] <= part
    assert same(rn.rn_kcp_hier(g, R, S, 2_000, rn.RN_INF, part), og.kcp(R, S, 2_000))


@pytest.mark.parametrize("part", [512, 4096])
def test_many_arcs_into_one_node(rn, oracle, part):
    """A node that hundreds of arcs of every part lead to: each source has as many routes to it,
    of which the least counts."""
    e = I.road_graph(8_000, 20_800, 231)
    rng = np.random.default_rng(232)
    t = rng.choice(np.arange(1, e.n), 5_000, replace=False)
    e = I.EdgeList(e.n, np.r_[e.src, e.dst, t].astype(np.uint32), np.r_[e.dst, e.src, np.zeros(len(t))].astype(np.uint32),
                   np.r_[e.w, e.w, rng.integers(1, 3_000, len(t))].astype(np.uint32), None, {})
    g = rn.rn_graph_load(e.src, e.dst, e.w, e.n, flags=rn.RN_REORDER)
    og = oracle.graph(e.n, e.src, e.dst, e.w, undirected=False)
    R, S = I.disjoint_sets(e.n, 600, 200, 233)
    for theta in (8_000, rn.RN_INF):
        ref = og.join(R, S, min(theta, rn.RN_THETA_MAX))
        assert same(rn.rn_distance_join_hier(g, R, S, theta, part), ref), theta
