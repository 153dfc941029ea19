"""Host-side rule of the 2D strip kernels (no GPU call): a small C++ program,
compiled with nvcc and linked against libjfnk.so, checks that a reducing call is
taken only where its partials fit the reduction scratch
(tests/host/strips_check.cu)."""
import os
import subprocess

import pytest

from test_host_tiling import ROOT, _nvcc


def test_reducing_calls_fit_the_scratch(tmp_path):
    from paper_2103_13890_gb300 import build as b
    if not os.path.exists(b.LIB):
        b.build()
    nvcc = _nvcc()
    if nvcc is None:
        pytest.skip("nvcc not found")
    libdir = os.path.dirname(b.LIB)
    exe = str(tmp_path / "strips_check")
    subprocess.run([nvcc, *b.ARCH, "-std=c++17", "-O1", "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_2103_13890_gb300", "csrc"),
                    os.path.join(ROOT, "tests", "host", "strips_check.cu"), "-o", exe,
                    "-L", libdir, "-ljfnk", "-Xlinker", "-rpath", "-Xlinker", libdir],
                   check=True, capture_output=True, text=True)
    out = subprocess.run([exe], capture_output=True, text=True)
    assert out.returncode == 0, out.stdout + out.stderr
    assert out.stdout.strip() == "ok 32"
