"""Registers and spills of kernels whose launch shape depends on them, as ptxas
reports them for sm_103a (no GPU)."""
import os
import re
import subprocess

from paper_2008_12820_gb300 import build as B


def resources(source, tmp_path):
    """{mangled kernel name: (registers, bytes of spill stores)} of a source"""
    r = subprocess.run([B.nvcc()] + B.ARCH + B.FLAGS + ["-Xptxas", "-v", "-c", os.path.join(B.SRC, source), "-o",
                       str(tmp_path / "out.o")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    found = re.findall(r"Compiling entry function '(\w+)'.*?(\d+) bytes spill stores.*?Used (\d+) registers", r.stdout +
                       r.stderr, re.S)
    return {name: (int(regs), int(spill)) for name, spill, regs in found}


def test_dot_products_run_in_one_wave(tmp_path):
    """Their grid is eight blocks of 256 threads per SM: 32 of the 65536 registers
    for each of 2048 threads."""
    k = {n: v for n, v in resources("vec.cu", tmp_path).items() if "k_reduce2" in n}
    assert len(k) >= 4
    assert all(regs <= 65536 // 2048 and spill == 0 for regs, spill in k.values()), k
