"""What follows a wait that a kernel gave up, in the bounds-checked build (librn_checks.so)."""
import ctypes
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def checks_lib():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1607_07696_gb300 import build as B

    return B.build(checks=True)


@pytest.mark.parametrize("n", [(1 << 15), (1 << 15) + 1, 100_003])
def test_passes_behind_a_failed_one_write_nothing(checks_lib, n):
    """A pass whose wait is cut leaves gaps in its output.  The passes behind it would scatter
    what is in the gaps by counts taken from other records, past the buffers' ends: they must
    find the failed check and write nothing."""
    f = ctypes.CDLL(checks_lib).rn_checks_sort_after_failure
    f.argtypes = [ctypes.c_uint64, ctypes.POINTER(ctypes.c_uint64)]
    changed = ctypes.c_uint64(1 << 60)
    assert f(n, ctypes.byref(changed)) == 0
    assert changed.value == 0


SCRIPT = r"""
import ctypes, sys
sys.path.insert(0, ROOT)
import numpy as np
from paper_1607_07696_gb300 import inputs as I, rn
fail = ctypes.CDLL(rn.LIB_PATH).rn_checks_fail_sort
e = I.road_graph(70_000, 194_000, 7)
g = rn.rn_graph_load(e.src, e.dst, e.w, e.n)
tiles = rn.rn_graph_load(e.src, e.dst, e.w, e.n, cfg={"tile_width": 32})
R, S = I.disjoint_sets(e.n, 3000, 4000, 8)
theta = int(20 * np.median(e.w))
calls = {  # result sizes of 2^15 pairs and more: their sorts take the single-launch passes
    "join": lambda: rn.rn_distance_join(tiles, R, S, theta),
    "kcp": lambda: rn.rn_kcp(g, R, S, 300_000),
    "kcp by tiles": lambda: rn.rn_kcp(tiles, R, S, 40_000),
    "join_many": lambda: rn.rn_join_many(tiles, [(R, S, theta), (S[:500], R, theta // 2)]),
    "hier join": lambda: rn.rn_distance_join_hier(g, R, S, theta, 1024),
    "hier kcp": lambda: rn.rn_kcp_hier(g, R, S, 50_000, rn.RN_INF, 1024),
    "batch": lambda: rn.rn_batch_run(rn.rn_batch_create([(g, R, S, theta), (g, S, R, theta // 2)])),
}
for name, call in calls.items():
    call()
    fail(1 << 20)
    call()
    sorts = (1 << 20) - fail(0)
    assert sorts >= 1, name
    for nth in range(1, sorts + 1):
        fail(nth)
        try:
            call()
            raise SystemExit(f"{name}: the failed wait of sort {nth} of {sorts} was not reported")
        except rn.RNError as ex:
            assert ex.status == rn.RN_EINTERNAL, (name, nth, ex)
        assert fail(0) == 0
    call()
    print(name, sorts)
print("reported")
"""


def test_failed_waits_are_reported(checks_lib):
    """Whatever sort of a call gives up a wait, the call ends with RN_EINTERNAL (and the next
    one is served)."""
    env = dict(os.environ, RN_LIBRARY=checks_lib)
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", "ROOT = %r\n" % root + SCRIPT], env=env, capture_output=True, text=True,
                       timeout=600)
    assert r.returncode == 0, (r.stdout + r.stderr)[-4000:]
    assert r.stdout.endswith("reported\n")
