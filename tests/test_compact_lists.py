"""Host-side checks of the gather lists of the compact and the wide FP32 kernels
(small C++ programs linked against the library); no GPU needed."""
import os
import shutil
import subprocess

import pytest

from paper_2301_09662_gb300 import build_lib

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def checkers(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    so = build_lib.build()
    libdir = os.path.dirname(so)
    out = {}
    for name in ("compact", "wide"):
        exe = str(tmp_path_factory.mktemp("lists") / f"{name}_lists_check")
        subprocess.run([nvcc, "-std=c++17", "-O2", "-I", os.path.join(ROOT, "include"),
                        "-I", os.path.join(ROOT, "paper_2301_09662_gb300", "csrc"),
                        os.path.join(ROOT, "tests", "native", f"{name}_lists_check.cu"),
                        "-o", exe, "-L", libdir, "-lepic", "-Xlinker", "-rpath=" + libdir],
                       check=True, capture_output=True)
        out[name] = exe
    return out


@pytest.mark.parametrize("A,K,span,C,P", [
    (256, 5, 49, 3, 2),     # LWA-like
    (256, 1, 45, 2, 2),     # point kernel (taper)
    (101, 3, 64, 2, 1),     # the widest aperture, single polarisation
    (1024, 7, 64, 1, 2),    # limits of the 16-bit entries
    (300, 5, 65, 1, 2),     # too wide: refused
    (64, 9, 40, 1, 2),      # K (K + 1) past the tap slots: refused
    (1, 3, 3, 1, 1),        # one footprint
])
def test_lists(checkers, A, K, span, C, P):
    r = subprocess.run([checkers["compact"], str(A), str(K), str(span), str(C), str(P)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.parametrize("A,K,sx,sy,C", [
    (2048, 7, 124, 124, 2),   # dense array
    (300, 5, 128, 128, 1),    # the widest aperture
    (300, 5, 129, 60, 1),     # too wide: refused
    (90, 3, 40, 65, 2),       # one row in the second band
    (60, 15, 30, 64, 1),      # widest kernel, one band exactly full
    (1, 1, 1, 1, 1),
])
def test_wide_lists(checkers, A, K, sx, sy, C):
    r = subprocess.run([checkers["wide"], str(A), str(K), str(sx), str(sy), str(C)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
