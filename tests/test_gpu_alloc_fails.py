"""Device allocations that fail in the middle of a call: the call ends with RN_ENOMEM (or does
without the memory), and the next one finds no buffer that is not there."""
import ctypes as C

import numpy as np
import pins
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


class Allocator:
    """Memory from torch; refuses the allocation that `refuse` names (by number or by size)."""

    def __init__(self, rn):
        import torch

        torch.cuda.init()
        self.rn, self.left, self.sizes, self.refused = rn, None, (), []

        def alloc(nbytes, ctx):
            if self.left is not None:
                self.left -= 1
            if self.left == 0 or int(nbytes) in self.sizes:
                self.refused.append(int(nbytes))
                return None
            p = torch.cuda.caching_allocator_alloc(int(nbytes), 0, torch.cuda.default_stream(0))
            torch.cuda.default_stream(0).synchronize()
            return p

        self.hook = (rn._ALLOC_FN(alloc), rn._FREE_FN(lambda p, ctx: torch.cuda.caching_allocator_delete(int(p))))

    def __enter__(self):
        rn = self.rn
        rn._check(rn.lib().rn_set_allocator(C.cast(self.hook[0], C.c_void_p), C.cast(self.hook[1], C.c_void_p), None))
        return self

    def __exit__(self, *exc):
        self.rn._check(self.rn.lib().rn_set_allocator(None, None, None))


@pytest.fixture(scope="module")
def world(oracle):
    e = I.road_graph(12_000, 33_200, 221)
    return e, oracle.graph(e.n, e.src, e.dst, e.w), int(np.median(e.w))


def same(got, ref):
    return len(got[0]) == len(ref) and all(
        np.array_equal(x, y.astype(x.dtype)) for x, y in zip(got, (ref.u, ref.v, ref.d)))


@pytest.mark.parametrize("kind", ["join", "join from S", "hashed", "kcp", "many", "points", "box"])
def test_every_allocation_fails_once(rn, world, kind):
    e, og, med = world
    R, S = I.disjoint_sets(e.n, 700, 900, 222)
    if kind == "points":
        pts = pins.random_points(np.random.default_rng(223), pins.least_weights(e), 900)
        R, S = pts[:400], pts[400:]
        ref, call = og.join_points(R, S, 12 * med), lambda g: rn.rn_distance_join_points(g, R, S, 12 * med)
    elif kind == "kcp":
        ref, call = og.kcp(R, S, 3_000), lambda g: rn.rn_kcp(g, R, S, 3_000)
    elif kind == "many":
        ref, call = og.join(R, S, 12 * med), lambda g: rn.rn_join_many(g, [(R, S, 12 * med), (S[:80], R, 5 * med)])[0]
    elif kind == "box":
        box = np.asarray((-1, -1, 2, 2), np.float32)
        ref, call = og.join(R, S, 12 * med), lambda g: rn.rn_distance_join_box(g, R, S, 12 * med, box)
    elif kind == "join from S":
        S = S[:200]
        ref, call = og.join(R, S, 12 * med), lambda g: rn.rn_distance_join(g, R, S, 12 * med)
    else:
        ref, call = og.join(R, S, 12 * med), lambda g: rn.rn_distance_join(g, R, S, 12 * med)
    flags = rn.RN_UNDIRECTED | (0 if kind == "hashed" else rn.RN_REORDER)
    with Allocator(rn) as a:
        failed = 0
        for nth in range(1, 200):
            g = rn.rn_graph_load(e.src, e.dst, e.w, e.n, flags=flags, xy=e.xy if kind == "box" else None)
            a.left, a.refused = nth, []
            try:
                assert same(call(g), ref), nth
            except rn.RNError as ex:
                assert ex.status == rn.RN_ENOMEM, (nth, ex)
                failed += 1
            a.left = None
            if not a.refused:
                break
            for run in range(2):
                assert same(call(g), ref), (nth, run)
        assert not a.refused and failed >= 5


def test_without_room_for_rows(rn, world, oracle):
    """The rows of the search by pages are extra memory (64 bytes a node and overflow row): graphs,
    points and batches for which they do not fit are answered by the hashed search."""
    e, og, med = world
    deg = np.bincount(np.r_[e.src, e.dst], minlength=e.n)  # (no loops or parallel edges)
    rows = int(((np.maximum(deg, 8) - 8 + 6) // 7).sum())
    R, S = I.disjoint_sets(e.n, 700, 900, 224)
    ref, refk = og.join(R, S, 12 * med), og.kcp(R, S, 3_000)
    pts = pins.random_points(np.random.default_rng(225), pins.least_weights(e), 900)
    refp = og.join_points(pts[:400], pts[400:], 12 * med)

    def answers(g):
        for run in range(2):
            assert same(rn.rn_distance_join(g, R, S, 12 * med), ref), run
            assert same(rn.rn_kcp(g, R, S, 3_000), refk), run
            assert same(rn.rn_distance_join_points(g, pts[:400], pts[400:], 12 * med), refp), run
            assert same(rn.rn_distance_join_hier(g, R, S, 12 * med, 2048), ref), run

    def batch(g):
        b = rn.rn_batch_create([(g, R, S, 12 * med), (g, S[:80], R, 5 * med)])
        for run in range(4):  # eager, laid out again, recorded, replayed
            rn.rn_batch_run(b)
            assert same(rn.rn_batch_pairs(b, 0), ref) and same(rn.rn_batch_pairs(b, 1), og.join(S[:80], R, 5 * med)), run

    with Allocator(rn) as a:
        a.sizes = (64 * (e.n + rows),)
        g = rn.rn_graph_load(e.src, e.dst, e.w, e.n)
        assert a.refused == [64 * (e.n + rows)]
        a.sizes = ()
        answers(g)
        batch(g)
        g = rn.rn_graph_load(e.src, e.dst, e.w, e.n)
        n = e.n + 900
        a.sizes, a.refused = (64 * (n + n // 4 + rows), 64 * (2 * e.n + 1 + 2 * rows)), []  # points', a batch's
        answers(g)
        batch(g)
        assert a.refused == list(a.sizes)


def test_every_allocation_of_a_batch_fails_once(rn, world):
    """Balls past the first maps, so that the batch is laid out again between its runs."""
    e, og, med = world
    R, S = I.disjoint_sets(e.n, 500, 600, 226)
    queries = [(R, S, 45 * med), (S[:90], R, 5 * med), (R[:200], S[:300], 20 * med)]
    refs = [og.join(*q) for q in queries]
    g = rn.rn_graph_load(e.src, e.dst, e.w, e.n)
    with Allocator(rn) as a:
        failed = 0
        for nth in range(1, 200):
            b = rn.rn_batch_create([(g, *q) for q in queries])
            a.left, a.refused = nth, []
            for run in range(4):  # eager, laid out again, recorded, replayed
                try:
                    rn.rn_batch_run(b)
                except rn.RNError as ex:
                    assert ex.status == rn.RN_ENOMEM, (nth, ex)
                    failed += 1
                    break
                assert all(same(rn.rn_batch_pairs(b, i), ref) for i, ref in enumerate(refs)), (nth, run)
            a.left = None
            if not a.refused:
                break
            for run in range(4):
                rn.rn_batch_run(b)
                assert all(same(rn.rn_batch_pairs(b, i), ref) for i, ref in enumerate(refs)), (nth, run)
        assert not a.refused and failed >= 8
