"""What the assembler reports of the GEMM kernels: those with 18 warps have 96 registers
a thread, and what does not fit would be spilled on the path of every tile."""
import os
import re

from paper_1911_07384_gb300 import build


def test_gemm_kernels_do_not_spill():
    build.build()
    with open(os.path.join(build.BUILD, "ptxas.log")) as f:
        log = f.read()
    entries = re.findall(r"Compiling entry function '(\w*6k_gemm\w*)'.*?(\d+) bytes spill stores, (\d+) bytes spill loads",
                         log, re.S)
    assert len(entries) >= 20
    assert [e for e in entries if e[1:] != ("0", "0")] == []
