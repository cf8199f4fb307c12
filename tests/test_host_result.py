"""Host results (rn_api.cpp) whose copy from the device fails, over fakes of the CUDA calls."""
import os
import shutil
import subprocess
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1607_07696_gb300", "csrc")


def test_failed_copies_give_their_block_back(tmp_path):
    cxx = shutil.which("g++")
    inc = "/usr/local/cuda/include"
    if not cxx or not os.path.exists(os.path.join(inc, "cuda_runtime.h")):
        pytest.skip("g++ or the CUDA headers are missing")
    so = str(tmp_path / "result_driver.so")
    cmd = [cxx, "-std=c++17", "-O1", "-fPIC", "-shared", "-Wl,-z,lazy", "-Wl,-Bsymbolic", "-I", os.path.join(ROOT, "include"),
           "-I", CSRC, "-I", inc, os.path.join(ROOT, "tests", "sanitize", "result_driver.cpp"),
           os.path.join(CSRC, "rn_api.cpp"), "-o", so]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-4000:]
    code = ("import ctypes, os; n = ctypes.c_int(); L = ctypes.CDLL(%r, mode=os.RTLD_LAZY); "
            "print(L.failed_results(ctypes.byref(n)), n.value, flush=True); os._exit(0)" % so)
    r = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True)
    assert r.stdout.split() == ["0", "1"], r.stdout + r.stderr[-2000:]
