"""The packed complex64 sweeps' work tables on the host: every (set, orbit)
item of a window step exactly once, with its strings' addresses."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    gxx = shutil.which("g++")
    cuda_inc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    if gxx is None or not os.path.exists(os.path.join(cuda_inc, "cuda_runtime.h")):
        pytest.skip("needs g++ and the CUDA headers")
    exe = str(tmp_path_factory.mktemp("packed_tables") / "packed_tables_driver")
    csrc = os.path.join(ROOT, "paper_2605_03123_gb300", "csrc")
    r = subprocess.run([gxx, "-O2", "-std=c++17", "-I", cuda_inc, "-I",
                        os.path.join(ROOT, "include"), "-I", csrc,
                        os.path.join(ROOT, "tests", "packed_tables_driver.cpp"),
                        os.path.join(csrc, "fs_host.cpp"), "-o", exe],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    return exe


@pytest.mark.parametrize("N,n", [(6, 3), (7, 1), (8, 8), (9, 0), (10, 5), (12, 6), (13, 7),
                                 (16, 3), (16, 8), (20, 3), (32, 1)])
@pytest.mark.parametrize("nk", [1, 2, 3, 7, 32, 64])
def test_items_once_each(driver, N, n, nk):
    out = subprocess.run([driver, str(N), str(n), str(nk)], capture_output=True, text=True)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout
