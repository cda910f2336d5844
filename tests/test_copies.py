"""The helper threads' copies of kept results (header-only C++): overlapping
destinations are written in order, every ticket is released once."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.mark.parametrize("threads", [0, 1, 4])
def test_copies_in_order(threads, tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    exe = tmp_path / "copies_check"
    subprocess.check_call([gxx, "-O2", "-std=c++17", "-pthread", "-I",
                           os.path.join(ROOT, "paper_2010_15879_gb300", "csrc"),
                           os.path.join(ROOT, "tests", "copies_check.cpp"), "-o", str(exe)])
    out = subprocess.run([str(exe), str(threads)], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, out.stdout + out.stderr
    assert out.stdout.startswith("ok")
