"""What the propagation calls copy to the device is still there when a copy that
the runtime puts off gets to it (a copy from pageable memory need not be staged).
The host code of the ABI runs here against a runtime of stand-ins."""
import os
import shutil
import subprocess

import pytest

from paper_2509_04666_gb300 import workloads as W

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2509_04666_gb300", "csrc")
CUDA = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")


def test_copies_outlive_the_host_arrays_of_the_call(tmp_path):
    if shutil.which("g++") is None or not os.path.isdir(CUDA):
        pytest.skip("no g++ or CUDA headers")
    exe, table = str(tmp_path / "uploads"), tmp_path / "table"
    # device symbols the calls below do not reach stay unresolved
    subprocess.run(["g++", "-x", "c++", "-std=c++17", "-O1", "-include", "math.h", "-I", CUDA, "-I", CSRC,
                    os.path.join(CSRC, "kete_abi.cu"), os.path.join(HERE, "host_uploads.cpp"), "-o", exe,
                    "-Wl,--unresolved-symbols=ignore-all"], check=True)
    table.write_bytes(W.static_sun_table(W.T0 - 20.0, W.T0 + 1000.0).to_bytes())
    # freed memory is overwritten at once
    out = subprocess.run([exe, str(table), repr(W.T0)], check=True, capture_output=True, text=True,
                         env={**os.environ, "MALLOC_PERTURB_": "165"}).stdout
    rc, stale, copies = map(int, out.split())
    assert rc == 0 and copies > 20
    assert stale == 0, (stale, copies)
