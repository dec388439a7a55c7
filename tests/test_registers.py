"""What the compiler says of kernels whose registers were once cut down behind the programmer's back (nvcc, no GPU).

A CTA of 1024 threads that has its SM to itself may use 64 registers a thread; without a word about it ptxas may decide for two CTAs an SM
and spill.
"""
import os
import re
import subprocess

import pytest

from paper_2601_17818_b200 import build


@pytest.mark.parametrize("source,kernel", [("filter.cu", "vic_finalize_kernelILi1ELi1E")])
def test_nothing_is_spilled(source, kernel, tmp_path):
    r = subprocess.run([build._nvcc(), *build.NVCC_FLAGS, "-Xptxas", "-v", "-cubin", os.path.join(build.CSRC, source), "-o", str(tmp_path / "x")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    said = re.findall(rf"Compiling entry function '\S*{kernel}.*?(\d+) bytes spill stores, (\d+) bytes spill loads.*?Used (\d+) registers",
                      r.stderr, re.S)
    assert said and all(stores == loads == "0" for stores, loads, _ in said), said
