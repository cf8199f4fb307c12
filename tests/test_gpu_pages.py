"""The source search by pages at the sizes where it can go wrong, against the oracle (integer
distances: equal or wrong).  Covered: balls of a few nodes up to thousands (one warp a source,
2 to 32 warps a source, maps that overflow), ids with and without locality (the hashed
search answers the latter), nodes whose arcs fill a row of eight slots exactly, go on in one or
several overflow rows, or are too many for the search by pages, and distances at the end of
the 31-bit range."""
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


@pytest.fixture(scope="module")
def oracle():
    from oracle import oracle as O

    return O.default()


def same(got, ref):
    return len(got[0]) == len(ref) and all(
        np.array_equal(x, y.astype(x.dtype)) for x, y in zip(got, (ref.u, ref.v, ref.d)))


@pytest.mark.parametrize("reorder", [True, False])
@pytest.mark.parametrize("ball", [1, 31, 300, 1100, 2600, 6000, 15000])
def test_ball_sizes(rn, oracle, ball, reorder):
    e = I.road_graph(40_000, 110_800, 91)
    flags = rn.RN_UNDIRECTED | (rn.RN_REORDER if reorder else 0)
    og = oracle.graph(e.n, e.src, e.dst, e.w)
    for nR, nS in ((7, 900), (3000, 4000)):
        if nR * ball > 2e7:
            continue
        R, S = I.disjoint_sets(e.n, nR, nS, 92 + nR)
        theta = int(np.sort(og.sssp(int(R[0]))[0])[ball])
        g = rn.rn_graph_load(e.src, e.dst, e.w, e.n, flags=flags, cfg={"tile_width": 1})
        ref = og.join(R, S, theta)
        for run in range(2):  # without, then with the balls of an earlier search
            assert same(rn.rn_distance_join(g, R, S, theta), ref), (nR, run)
        k = max(1, len(ref) // 3)
        assert same(rn.rn_kcp(g, R, S, k, theta), og.kcp(R, S, k, theta)), nR
        outs = rn.rn_join_many(g, [(R, S, theta), (S[:50], R, theta // 2)])
        assert same(outs[0], ref) and same(outs[1], og.join(S[:50], R, theta // 2)), nR


def hub_graph(degree: int, wmax: int = 50):
    """Nodes in a line, and nodes of the given degree joined to their neighbourhood."""
    n = 800
    rng = np.random.default_rng(degree)
    edges = {(i, i + 1): int(rng.integers(1, wmax)) for i in range(n - 1)}
    for hub in (100, 400, 401, 700):
        for other in rng.permutation(np.r_[hub - 90:hub, hub + 1:hub + 90])[:max(0, degree - 2)]:
            edges[(min(hub, int(other)), max(hub, int(other)))] = int(rng.integers(1, wmax))
    e = np.array(list(edges), np.int64)
    return n, e[:, 0], e[:, 1], np.array(list(edges.values()), np.int64)


@pytest.mark.parametrize("degree", [7, 8, 9, 14, 15, 16, 22, 23, 50, 64, 90])
def test_row_overflow(rn, oracle, degree):
    n, src, dst, w = hub_graph(degree)
    og = oracle.graph(n, src, dst, w)
    R, S = I.disjoint_sets(n, 150, 250, degree)
    rng = np.random.default_rng(degree)
    i = rng.integers(0, len(w), size=120)
    pts = np.stack([src[i], dst[i], (rng.random(120) * (w[i] + 1)).astype(np.int64)], axis=1)
    for flags in (rn.RN_UNDIRECTED, rn.RN_UNDIRECTED | rn.RN_REORDER):
        g = rn.rn_graph_load(src, dst, w, n, flags=flags, cfg={"leaf_size": 64})
        for theta in (0, 40, 400, rn.RN_INF):
            ref = og.join(R, S, min(theta, rn.RN_THETA_MAX))
            assert same(rn.rn_distance_join(g, R, S, theta), ref), (flags, theta)
        assert same(rn.rn_distance_join_points(g, pts[:60], pts[60:], 200), og.join_points(pts[:60], pts[60:], 200)), flags
        assert same(rn.rn_distance_join_hier(g, R, S, 400, 64), og.join(R, S, 400)), flags
        b = rn.rn_batch_create([(g, R, S, 400), (g, S[:70], R, 90)])
        for _ in range(3):
            rn.rn_batch_run(b)
            assert same(rn.rn_batch_pairs(b, 0), og.join(R, S, 400)), flags
            assert same(rn.rn_batch_pairs(b, 1), og.join(S[:70], R, 90)), flags


@pytest.mark.parametrize("theta", [(1 << 31) - 3, (1 << 31) - 2, (1 << 31) - 1, 1 << 31, 0xFFFFFFFF])
def test_longest_distances(rn, oracle, theta):
    """A path whose distances reach past 2^31: the search by pages holds them up to 2^31 - 2,
    and larger bounds are answered by the searches that hold 32 bits."""
    w = np.full(199, (1 << 24) - 1, np.int64)
    w[40:104] = 1 << 23  # sums that hit 2^31 closely
    e = I.path_graph(w)
    og = oracle.graph(e.n, e.src, e.dst, e.w)
    ids = np.random.default_rng(5).permutation(e.n)
    R, S = ids[:80], ids[80:]
    for T in (0, 1):
        g = rn.rn_graph_load(e.src, e.dst, e.w, e.n, cfg={"tile_width": T})
        ref = og.join(R, S, min(theta, rn.RN_THETA_MAX))
        assert same(rn.rn_distance_join(g, R, S, theta), ref), T
        assert same(rn.rn_kcp(g, R, S, 500, theta), og.kcp(R, S, 500, min(theta, rn.RN_THETA_MAX))), T


@pytest.mark.parametrize("k,paged", [(5, True), (8, True), (10, False), (16, False)])
def test_dense_graphs(rn, oracle, k, paged):
    """Planar graphs around the most overflow rows a node that the search by pages takes (three to
    four nodes): rows are held, 64 bytes a node and overflow row, where it does."""
    rng = np.random.default_rng(k)
    xy = rng.random((12_000, 2))
    ab = I._knn_edges(I._knn_table(xy, k), k)
    w = rng.integers(1, 300, size=len(ab))
    deg = np.bincount(ab.ravel(), minlength=len(xy))
    rows = int(((np.maximum(deg, 8) - 8 + 6) // 7).sum())
    assert (4 * rows <= 3 * len(xy)) == paged
    og = oracle.graph(len(xy), ab[:, 0], ab[:, 1], w)
    g, plain = (rn.rn_graph_load(ab[:, 0], ab[:, 1], w, len(xy), flags=rn.RN_UNDIRECTED | f) for f in (rn.RN_REORDER, 0))
    held = rn.rn_graph_info(g)["device_bytes"] - rn.rn_graph_info(plain)["device_bytes"]
    assert held == (64 * (len(xy) + rows) if paged else 0)
    R, S = I.disjoint_sets(len(xy), 700, 900, k)
    for theta in (150, 700):
        ref = og.join(R, S, theta)
        for run in range(2):
            assert same(rn.rn_distance_join(g, R, S, theta), ref), (theta, run)
    assert same(rn.rn_kcp(g, R, S, 3_000), og.kcp(R, S, 3_000))
