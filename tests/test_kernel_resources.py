"""Registers of kernels whose speed rests on how many CTAs an SM holds, as ptxas reports them."""
import re
import subprocess

from paper_2608_17402_gb300 import _build


def _registers(source):
    """{mangled kernel name: registers a thread} of one source file."""
    cmd = [_build._nvcc(), *_build.ARCH, "-O3", "-std=c++17", "-I", _build.INCLUDE, "-I", _build.CSRC,
           "--expt-relaxed-constexpr", "-Xptxas", "-v", "-cubin", "-o", "/dev/null", f"{_build.CSRC}/{source}"]
    out = subprocess.run(cmd, capture_output=True, text=True, check=True).stderr
    return {n: int(r) for n, r in re.findall(r"Compiling entry function '(\S+)'.*?Used (\d+) registers", out, re.S)}


def test_gates_leave_room_for_four_ctas():
    """65536 registers an SM, 256 threads a CTA: 64 a thread let four CTAs in."""
    regs = {n: r for n, r in _registers("backward.cu").items() if "bwd_gates" in n}
    assert regs
    assert max(regs.values()) <= 64, regs
