"""What a search teaches the next ones about ball sizes: queries whose balls fit the source search
stay with it (tile_width 1 in their statistics) whatever was searched before, and equal the oracle."""
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


@pytest.fixture(scope="module")
def world():
    """A road-like graph of 100,000 nodes and 300 pairs of nodes joined to nothing else."""
    from oracle import oracle as O

    e = I.road_graph(100_000, 277_000, 201)
    a = np.arange(300) * 2 + e.n
    e = I.EdgeList(e.n + 600, np.r_[e.src, a].astype(np.uint32), np.r_[e.dst, a + 1].astype(np.uint32),
                   np.r_[e.w, np.full(300, 7)].astype(np.uint32), None, {})
    return e, O.default().graph(e.n, e.src, e.dst, e.w)


def sets(e, rng, nR, nS, alone):
    """R and S, with the first node of `alone` of the pairs in R."""
    main = rng.permutation(e.n - 600)[:nR + nS - alone].astype(np.uint32)
    pairs = (e.n - 600 + 2 * rng.permutation(300)[:alone]).astype(np.uint32)
    return np.r_[pairs, main[:nR - alone]], main[nR - alone:]


@pytest.mark.parametrize("reorder,ball", [(True, 6000), (False, 4000)])
def test_after_a_first_search_that_few_sources_complete(rn, world, reorder, ball):
    """The first search of a workspace has maps for balls of about 2,000 nodes: only the sources in
    the pairs complete it.  Their two nodes are not the mean ball."""
    e, og = world
    rng = np.random.default_rng(202)
    R, S = sets(e, rng, 300, 400, 40)
    theta = int(np.sort(og.sssp(int(R[-1]))[0])[ball])
    g = rn.rn_graph_load(e.src, e.dst, e.w, e.n, flags=rn.RN_UNDIRECTED | (rn.RN_REORDER if reorder else 0))
    assert same(rn.rn_distance_join(g, R, S, theta), og.join(R, S, theta))
    assert rn.rn_last_query_stats()["retried_tiles"] > 200
    # balls of about 1,900 nodes hold the k closest pairs
    assert same(rn.rn_kcp(g, R, S, 2_000), og.kcp(R, S, 2_000))
    st = rn.rn_last_query_stats()
    assert st["tile_width"] == 1 and st["passes"] <= 2
    assert st["slots"] < 300 * 3 * ball


@pytest.mark.parametrize("reorder,ball", [(True, 6000), (False, 4000)])
def test_after_joins_of_several_bounds(rn, world, reorder, ball):
    """Joins searched together, most of them with a small bound: their mean ball is not the one at
    the largest bound."""
    e, og = world
    rng = np.random.default_rng(203)
    R, S = sets(e, rng, 300, 400, 0)
    theta = int(np.sort(og.sssp(int(R[-1]))[0])[ball])
    small = int(np.sort(og.sssp(int(R[-1]))[0])[3])
    P, Q = sets(e, rng, 4000, 4000, 0)
    g = rn.rn_graph_load(e.src, e.dst, e.w, e.n, flags=rn.RN_UNDIRECTED | (rn.RN_REORDER if reorder else 0))
    for run in range(2):
        outs = rn.rn_join_many(g, [(P, Q, small), (R, S, theta)])
        assert same(outs[0], og.join(P, Q, small)) and same(outs[1], og.join(R, S, theta)), run
    assert same(rn.rn_kcp(g, R, S, 2_000), og.kcp(R, S, 2_000))
    st = rn.rn_last_query_stats()
    assert st["tile_width"] == 1 and st["passes"] <= 2
    assert st["slots"] < 300 * 3 * ball
