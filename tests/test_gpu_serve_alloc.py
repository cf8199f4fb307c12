"""A server's requests within the sizes its workers are reserved for allocate no device memory:
an allocation may wait for every stream's work, and the free that follows a growth does."""
import ctypes as C
import threading

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


def test_requests_allocate_nothing(rn, oracle):
    import torch

    made, lock = [], threading.Lock()

    def alloc(nbytes, ctx):
        p = torch.cuda.caching_allocator_alloc(int(nbytes), 0, torch.cuda.default_stream(0))
        torch.cuda.default_stream(0).synchronize()
        with lock:
            made.append(int(nbytes))
        return p

    hook = (rn._ALLOC_FN(alloc), rn._FREE_FN(lambda p, ctx: torch.cuda.caching_allocator_delete(int(p))))
    torch.cuda.init()
    e = I.road_graph(60_000, 166_000, 211)
    og = oracle.graph(e.n, e.src, e.dst, e.w)
    med = int(np.median(e.w))
    requests = []
    for i in range(60):  # joins from R and from S, alone and grouped, k closest pairs of all sizes
        rng = np.random.default_rng(i)
        nR, nS = (int(x) for x in rng.integers(20, 3000, size=2))
        R, S = I.disjoint_sets(e.n, nR, nS, 300 + i)
        if i % 5 == 4:  # (balls of up to about 1,500 nodes: past 20,000, a search takes maps in device memory)
            k = max(1, min(int(rng.integers(1, 20_000)), nR * nS * 1_500 // e.n))
            requests.append((R, S, rn.RN_INF, k))
        else:
            requests.append((R, S, int(rng.integers(3, 20)) * med, 0))
    rn._check(rn.lib().rn_set_allocator(C.cast(hook[0], C.c_void_p), C.cast(hook[1], C.c_void_p), None))
    try:
        g = rn.rn_graph_load(e.src, e.dst, e.w, e.n)
        srv = rn.rn_serve_create(g, slab_bytes=1 << 30, workers=4)
        made.clear()
        for rounds in range(2):  # one after another, then all at once
            if rounds:
                tickets = [rn.rn_serve_submit(srv, *q) for q in requests]
                results = [rn.rn_serve_wait(srv, t) for t in tickets]
            else:
                results = [rn.rn_serve_wait(srv, rn.rn_serve_submit(srv, *q)) for q in requests]
            assert made == []
            for (R, S, theta, k), got in list(zip(requests, results))[::9]:
                ref = og.kcp(R, S, k) if k else og.join(R, S, theta)
                assert len(got[0]) == len(ref) and all(
                    np.array_equal(x, y.astype(x.dtype)) for x, y in zip(got, (ref.u, ref.v, ref.d)))
        srv.close()
        del srv, g
    finally:
        rn._check(rn.lib().rn_set_allocator(None, None, None))
