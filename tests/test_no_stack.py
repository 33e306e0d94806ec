"""No kernel keeps anything in local memory: a stack frame is a copy of parameters or an array that the compiler could not keep
in registers, and costs a bandwidth-bound kernel up to half its rate.  (What the assembler reports; no device is needed.)"""
import os
import re
import subprocess

import pytest

from paper_2506_19651_b200 import build as pbuild


@pytest.mark.parametrize("source", ["assemble_kernel.cu", "merge_kernel.cu", "decode_kernel.cu", "attn_kernel.cu"])
def test_no_stack_frame(source, tmp_path):
    r = subprocess.run([pbuild._nvcc(), *pbuild.NVCC_FLAGS[:2], "-O3", "-std=c++17", "-Xptxas", "-v", "-cubin",
                        os.path.join(pbuild.CSRC, source), "-o", str(tmp_path / "x")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    frames = re.findall(r"(\d+) bytes stack frame, (\d+) bytes spill stores", r.stderr)
    assert frames and all(f == ("0", "0") for f in frames), r.stderr
