"""The shared-memory layout of the row sweep (csrc/hm_row.cuh) on the host: no table starts below its alignment."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_tables_start_on_their_alignment(tmp_path):
    from paper_0706_3293_gb300 import build
    try:
        nvcc = build.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    exe = str(tmp_path / "row_align_check")
    subprocess.check_call([nvcc] + build.ARCH + ["-std=c++17", "--expt-relaxed-constexpr", "-I", build.CSRC, "-I",
                                                 os.path.join(ROOT, "include"), "-o", exe,
                                                 os.path.join(ROOT, "tests", "native", "row_align_check.cu")])
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
