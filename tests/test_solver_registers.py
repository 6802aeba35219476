"""The plain solver kernel, which runs every batch, keeps its values in registers:
the compiler's report (`-Xptxas -v`) names no spills at any block size.  A spilled
value is read back from local memory after every team barrier (the barrier's
acquire drops L1)."""
import os
import re
import subprocess

import pytest

from paper_2309_14584_gb300 import build as B


def test_plain_variant_does_not_spill(tmp_path):
    try:
        cc = B.nvcc()
    except RuntimeError:
        pytest.skip("nvcc not found")
    flags = B.ARCH + ["-O3", "-lineinfo", "-std=c++17", "-static-global-template-stub=false", "-I", B.INCLUDE, "-I",
                      B.CSRC, "-Xptxas", "-v"]
    procs = {bt: subprocess.Popen([cc] + flags + ["-cubin", os.path.join(B.CSRC, f"fct_solve_k{bt}.cu"), "-o",
                                                  str(tmp_path / f"k{bt}.cubin")],
                                  stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
             for bt in (128, 256, 512)}
    for bt, p in procs.items():
        out, _ = p.communicate()
        assert p.returncode == 0, out
        # fct_solve_kernel<bt, SV = false, DEEP = 0, ...>
        found = re.findall(r"fct_solve_kernelILi\d+ELb0ELi0E\w*\n\s*(\d+) bytes stack frame, (\d+) bytes spill "
                           r"stores, (\d+) bytes spill loads", out)
        assert found == [("0", "0", "0")], (bt, found)
