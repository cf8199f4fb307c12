"""The ordering of a join's pairs at the sizes where its kernels change over, against the oracle:
the placement's and the rank order's longest segment (256 pairs), the radix sort's change to
one launch per digit (2^18 records, and a last tile of one), and a placement of many blocks."""
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
def world():
    """A connected graph (the largest component of a road-like one): unbounded joins pair all."""
    import scipy.sparse as sp
    from scipy.sparse.csgraph import connected_components

    from oracle import oracle as O

    e = I.road_graph(6000, 16620, 131)
    _, comp = connected_components(sp.coo_matrix((np.ones(e.m), (e.src, e.dst)), shape=(e.n, e.n)), directed=False)
    big = np.nonzero(comp == np.bincount(comp).argmax())[0]
    return e, O.default().graph(e.n, e.src, e.dst, e.w), np.random.default_rng(132).permutation(big)


def same(got, ref):
    return len(got[0]) == len(ref) and all(
        np.array_equal(x, y.astype(x.dtype)) for x, y in zip(got, (ref.u, ref.v, ref.d)))


@pytest.mark.parametrize("nR,nS", [
    (900, 1), (900, 31), (900, 255), (900, 256), (900, 257),  # searched from S: up to nS pairs of one u
    (40, 256), (40, 257), (1, 3000), (3000, 1),               # searched from R, from one source
    (512, 511), (512, 512), (513, 512),                       # 2^18 records and around
    (512, 520), (577, 641),                                   # ragged last tiles of the sort
    (4100, 900),                                              # 3.7 million
])
def test_every_pair(rn, world, nR, nS):
    e, og, nodes = world
    R, S = nodes[:nR], nodes[nR:nR + nS]
    g = rn.rn_graph_load(e.src, e.dst, e.w, e.n)
    ref = og.join(R, S, rn.RN_THETA_MAX)
    assert len(ref) == nR * nS
    for run in range(2):
        assert same(rn.rn_distance_join(g, R, S, rn.RN_INF), ref), run
    k = min(len(ref), 300_000)
    o = np.lexsort((ref.v, ref.u, ref.d))[:k]
    u, v, d = rn.rn_kcp(g, R, S, k)
    assert np.array_equal(u, ref.u[o]) and np.array_equal(v, ref.v[o]) and np.array_equal(d, ref.d[o].astype(d.dtype))


def test_many_placement_blocks(rn, world):
    e, og, nodes = world
    R, S = nodes[:5300], nodes[5300:5700]  # 83 blocks of 64 segments, some of them empty
    g = rn.rn_graph_load(e.src, e.dst, e.w, e.n, cfg={"search_from": 1})
    for theta in (0, 9_000, 40_000):
        ref = og.join(R, S, theta)
        for run in range(2):
            assert same(rn.rn_distance_join(g, R, S, theta), ref), (theta, run)
