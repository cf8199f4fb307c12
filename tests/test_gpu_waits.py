"""What follows a wait that a kernel gave up, in the bounds-checked build (librn_checks.so)."""
import ctypes

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
