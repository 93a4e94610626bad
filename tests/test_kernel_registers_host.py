"""Registers of the SINT4 GEMM's instances, as ptxas reports them: the split among its warps takes no more than every instance is launched with."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = os.path.join(ROOT, "paper_2604_18117_b200", "csrc", "lq_gemm.cu")


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="nvcc not found")
@pytest.mark.parametrize("flags", [[], ["-DLQ_TIMELINE"]], ids=["plain", "timeline"])
def test_every_instance_is_launched_with_the_registers_that_its_warps_share(tmp_path, flags):
    r = subprocess.run(["nvcc", "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-Xcompiler", "-fPIC", "-Xptxas", "-v", *flags,
                        "-I", os.path.join(ROOT, "include"), "-I", os.path.dirname(SOURCE), "-c", SOURCE, "-o", str(tmp_path / "g.o")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    used = re.findall(r"Compiling entry function '\S*lq_gemm_kernel\S*' for[^\n]*\n(?:(?!Compiling)[^\n]*\n)*?[^\n]*Used (\d+) registers", r.stderr)
    with open(SOURCE) as f:
        lean, drain = map(int, re.search(r"LEAN_REGS = (\d+), DRAIN_REGS = (\d+);", f.read()).groups())
    assert len(used) == 9
    assert all(4 * lean + 8 * drain <= 12 * int(n) for n in used), used
