"""Kernels that stream from memory run as fast as the warps that an SM holds let
them: the registers that their full occupancy allows (65,536 of an SM over its
2,048 threads), as the assembler reports them."""
import os
import re
import subprocess

import pytest

from helpers import ROOT
from paper_2608_10139_gb300 import build


def _registers(source):
    """Registers by kernel (as named in the mangled entry) of one source file."""
    cmd = [build.nvcc()] + build.ARCH + build.FLAGS + ["-Xptxas", "-v", "-c", os.path.join(build.CSRC, source), "-o", os.devnull]
    r = subprocess.run(cmd, capture_output=True, text=True, cwd=ROOT)
    assert r.returncode == 0, r.stderr
    found = re.findall(r"Compiling entry function '(\S+)'.*?Used (\d+) registers", r.stderr, flags=re.S)
    assert found
    return {name: int(n) for name, n in found}


@pytest.mark.parametrize("source,kernels", [
    ("prefill.cu", ["k_embed"]),
    ("relational.cu", ["k_predicate_colsILi0ELi1E", "k_predicate_colsILi0ELi2E", "k_predicate_colsILi1ELi0E"]),
])
def test_streaming_kernels_fill_an_sm(source, kernels):
    registers = _registers(source)
    for kernel in kernels:
        of = {k: n for k, n in registers.items() if kernel in k}
        assert of and all(n <= 32 for n in of.values()), of
