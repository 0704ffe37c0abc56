"""Staging rows of voltages by words reads nothing outside the caller's block (no GPU: the address arithmetic)."""
import os
import shutil
import subprocess

import pytest

from test_host_logic import CSRC, ROOT, _cuda_include


def test_words_of_rows_stay_in_the_block(tmp_path):
    cxx, inc = shutil.which("g++") or shutil.which("c++"), _cuda_include()
    if not cxx or not inc:
        pytest.skip("host C++ compiler or CUDA headers not available")
    exe = str(tmp_path / "voltage_words")
    r = subprocess.run([cxx, "-O1", "-std=c++17", "-I", inc, "-I", CSRC,
                        os.path.join(ROOT, "tests", "host_voltage_words.cpp"), "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-3000:]
    out = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert out.stdout.split() == ["0", "0"]
