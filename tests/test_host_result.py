"""Host results (rn_api.cpp) and their page-locked blocks, over fakes of the CUDA calls."""
import os
import shutil
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1607_07696_gb300", "csrc")


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    cxx = shutil.which("g++")
    inc = "/usr/local/cuda/include"
    if not cxx or not os.path.exists(os.path.join(inc, "cuda_runtime.h")):
        pytest.skip("g++ or the CUDA headers are missing")
    so = str(tmp_path_factory.mktemp("result") / "result_driver.so")
    cmd = [cxx, "-std=c++17", "-O1", "-fPIC", "-shared", "-Wl,-z,lazy", "-Wl,-Bsymbolic", "-I", os.path.join(ROOT, "include"),
           "-I", CSRC, "-I", inc, os.path.join(ROOT, "tests", "sanitize", "result_driver.cpp"),
           os.path.join(CSRC, "rn_api.cpp"), "-o", so]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-4000:]
    return so


def run(so, call):
    code = ("import ctypes, os; n = ctypes.c_int(); L = ctypes.CDLL(%r, mode=os.RTLD_LAZY); print(%s, flush=True); "
            "os._exit(0)" % (so, call))
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    return r.stdout.split()


def test_failed_copies_give_their_block_back(driver):
    assert run(driver, "L.failed_results(ctypes.byref(n)), n.value") == ["0", "1"]


@pytest.mark.parametrize("n", [0, 1, 100, 2730, 2731, 5461, 5462, 8192, 100_000])
def test_blocks_are_used_again(driver, n):
    """Also by results far smaller than the smallest block (64 KB: 5,461 pairs)."""
    assert run(driver, f"L.blocks_for_results(ctypes.c_uint64({n}), 5)") == ["1"]
