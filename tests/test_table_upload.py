"""Tables that a plan needs together are uploaded together: after a failed allocation or copy the plan holds none
of them (no GPU: the CUDA runtime's calls are stand-ins)."""
import os
import shutil
import subprocess

import pytest

from test_host_logic import CSRC, ROOT, _cuda_include


def test_a_failed_upload_leaves_no_table_behind(tmp_path):
    cxx, inc = shutil.which("g++") or shutil.which("c++"), _cuda_include()
    if not cxx or not inc:
        pytest.skip("host C++ compiler or CUDA headers not available")
    exe = str(tmp_path / "table_upload")
    # upload() itself is not called here, so the CUDA runtime is not linked
    r = subprocess.run([cxx, "-O1", "-std=c++17", "-I", inc, "-I", CSRC,
                        os.path.join(ROOT, "tests", "host_table_upload.cpp"), "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    out = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0, out.stderr
    rows = [tuple(map(int, line.split())) for line in out.stdout.splitlines()]
    # three allocations and two copies (an empty table has nothing to copy): each may fail
    assert rows == [(0, 0, 0, 0, 20)] * 5 + [(1, 3, 3, 1, 20)]
