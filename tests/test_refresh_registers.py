"""The chunked refresh kernels keep everything in registers: what the assembler reports for each of them, compiled as the library is."""
import os
import re
import shutil
import subprocess

import pytest

from paper_2608_30386_b200 import build


@pytest.mark.skipif(not (shutil.which("nvcc") or os.path.exists(build._nvcc())), reason="no nvcc")
def test_no_chunked_kernel_spills(tmp_path):
    out = subprocess.run([build._nvcc(), *build.NVCC_FLAGS, "-Xptxas=-v", "-I", os.path.join(build.ROOT, "include"), "-I", build.CSRC,
                          "-c", os.path.join(build.CSRC, "refresh_chunked.cu"), "-o", str(tmp_path / "refresh_chunked.o")],
                         capture_output=True, text=True, check=True).stderr
    # per kernel: its name, then its stack frame and spills
    found = re.findall(r"Function properties for (\w*refresh_chunked_kernel\w*)\n"
                       r"\s*(\d+) bytes stack frame, (\d+) bytes spill stores, (\d+) bytes spill loads", out)
    assert len(found) == len(set(re.findall(r"Compiling entry function '(\w*refresh_chunked_kernel\w*)'", out))) > 0
    assert [f for f in found if f[1:] != ("0", "0", "0")] == []
