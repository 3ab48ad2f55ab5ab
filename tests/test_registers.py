"""Registers by the assembler's own report.  Of the residue GEMM the epilogue keeps 64 running values a thread in a budget of 96
registers, and a variant that spills more than a few of its addresses loses several percent."""
import os
import re
import shutil
import subprocess

import pytest

from paper_2609_09095_b200 import build as ozbuild


def _spills(unit, kernel, tmp_path):
    """Bytes of spill stores of every variant of a kernel."""
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    if shutil.which(nvcc) is None:
        pytest.skip("no nvcc")
    out = subprocess.run([nvcc, *ozbuild.NVCC_FLAGS, "-Xptxas=-v", "-c", os.path.join(ozbuild.CSRC, unit), "-o", str(tmp_path / "x.o")],
                         capture_output=True, text=True, check=True).stderr
    return {name: int(n) for name, n in re.findall(r"Function properties for (\S+)\n\s+\d+ bytes stack frame, (\d+) bytes spill stores", out)
            if kernel in name}


def test_residue_gemm_variants_spill_little(tmp_path):
    spills = _spills("oz_gemm_sm100.cu", "residue_gemm_kernel", tmp_path)
    assert len(spills) >= 30
    assert {name: n for name, n in spills.items() if n > 64} == {}
    native = {name: n for name, n in spills.items() if "residue_gemm_kernelILi1ELi1ELi1ELb1E" in name}
    assert len(native) >= 2 and set(native.values()) == {0}       # (packed before they are stored, the public one spilled 56 bytes and was 12 percent slower)


def test_reconstruction_variants_spill_little(tmp_path):
    """Four rows a thread keep numbers, sums and old values of C in 64 registers; what only some results need is out of line."""
    spills = _spills("oz_reconstruct.cu", "reconstruct_tiled_kernel", tmp_path)
    assert len(spills) == 36
    assert {name: n for name, n in spills.items() if n > 36} == {}
