"""Kernels whose comment says that their working set stays in registers: no spills in the compiler's report."""
import os
import re
import subprocess

import pytest


@pytest.mark.parametrize("source,kernel", [("eval.cu", "k_lm_solve"), ("inverse.cu", "k_trtri_tc")])
def test_no_spills(source, kernel, tmp_path):
    from paper_2509_26222_gb300 import build as B
    try:
        cc = B.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    r = subprocess.run([cc, *B.ARCH, "-O3", "-std=c++17", "-Xptxas", "-v", "-I", B.INC, "-cubin", "-o",
                        str(tmp_path / "k.cubin"), os.path.join(B.CSRC, source)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    found = re.findall(r"Compiling entry function '(\S+)'.*?\n.*?\n\s*\d+ bytes stack frame, (\d+) bytes spill stores",
                       r.stdout + r.stderr)
    spills = [int(n) for name, n in found if kernel in name]
    assert spills and max(spills) == 0
