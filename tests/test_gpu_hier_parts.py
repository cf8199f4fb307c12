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
