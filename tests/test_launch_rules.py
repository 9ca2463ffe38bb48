"""Host-side checks of the rules that choose launch shapes (a small C++ program
linked against the library); no GPU needed."""
import os
import shutil
import subprocess

import pytest

from paper_2301_09662_gb300 import build_lib

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_launch_rules(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    so = build_lib.build()
    libdir = os.path.dirname(so)
    exe = str(tmp_path / "launch_rules_check")
    subprocess.run([nvcc, "-std=c++17", "-O2", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_2301_09662_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "native", "launch_rules_check.cu"),
                    "-o", exe, "-L", libdir, "-lepic", "-Xlinker", "-rpath=" + libdir],
                   check=True, capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
