"""Registers of the residue GEMM by the assembler's own report: the epilogue keeps 64 running values a thread in a budget of 96
registers, and a variant that spills more than a few of its addresses loses several percent."""
import os
import re
import shutil
import subprocess

import pytest

from paper_2609_09095_b200 import build as ozbuild


def test_residue_gemm_variants_spill_little(tmp_path):
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    if shutil.which(nvcc) is None:
        pytest.skip("no nvcc")
    out = subprocess.run([nvcc, *ozbuild.NVCC_FLAGS, "-Xptxas=-v", "-c", os.path.join(ozbuild.CSRC, "oz_gemm_sm100.cu"), "-o", str(tmp_path / "x.o")],
                         capture_output=True, text=True, check=True).stderr
    spills = {name: int(n) for name, n in re.findall(r"Function properties for (\S+)\n\s+\d+ bytes stack frame, (\d+) bytes spill stores", out)
              if "residue_gemm_kernel" in name}
    assert len(spills) >= 30
    assert {name: n for name, n in spills.items() if n > 64} == {}
