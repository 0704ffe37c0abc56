"""After a bounded wait that ran out, the flag and the counts of split work items are cleared together (no GPU: the CUDA
runtime's calls are stand-ins)."""
import os
import shutil
import subprocess

import pytest

from test_host_logic import CSRC, ROOT, _cuda_include


def test_flag_and_counts_are_cleared_together(tmp_path):
    cxx, inc = shutil.which("g++") or shutil.which("c++"), _cuda_include()
    if not cxx or not inc:
        pytest.skip("host C++ compiler or CUDA headers not available")
    exe = str(tmp_path / "wait_flag")
    r = subprocess.run([cxx, "-O1", "-std=c++17", "-I", inc, "-I", CSRC, os.path.join(ROOT, "tests", "host_wait_flag.cpp"),
                        "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    out = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0, out.stderr
    assert out.stdout.split("\n")[:5] == [
        "1 0 0 2 0 5 0",     # no flag: a running integration's counts stay
        "1 0 0 2 0 5 0",
        "1 1 0 2 0 5 1",     # flag, a plan without split items
        "1 1 0 0 0 0 1",     # flag: both cleared, and waited for
        "1 0",               # a plan without a flag
    ]
