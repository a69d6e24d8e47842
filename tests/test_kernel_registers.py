"""Spills of the register-streaming GEMM, from the compiler's own report (nvcc, no GPU needed)."""
import os
import re
import shutil
import subprocess

import pytest

from paper_2504_05598_b200 import build


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="needs nvcc")
def test_one_row_variants_do_not_spill(tmp_path):
    """rowgemm_kernel<1, 8, LMHEAD, 8> runs once per drafted token, the one-row layer GEMMs four times per layer: they fill the 128
    registers that two CTAs per SM leave, and a value more goes to local memory."""
    out = subprocess.run(["nvcc", "-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-Xptxas", "-v",
                          "-c", os.path.join(build.CSRC, "rowgemm.cu"), "-o", str(tmp_path / "rowgemm.o")],
                         capture_output=True, text=True, check=True).stderr
    spills = {}
    for name, st, ld in re.findall(r"entry function '(\S+)'.*?(\d+) bytes spill stores, (\d+) bytes spill loads", out, re.S):
        m = re.search(r"rowgemm_kernelILi(\d+)ELi(\d+)ELi(\d+)ELi(\d+)EE", name)
        spills[tuple(map(int, m.groups()))] = (int(st), int(ld))
    one_row = {k: v for k, v in spills.items() if k[0] == 1}
    assert len(one_row) == 6 and all(v == (0, 0) for v in one_row.values()), one_row
