"""Kernels of a decode step and of a prompt pass keep their values in registers: what ptxas reports when it compiles them."""
import os
import re
import subprocess

import pytest

from paper_2404_08698_b200 import build as b


@pytest.mark.parametrize("source", ["attn_dec.cu", "attn_pf.cu", "gemm_cl.cu", "gemm_pf.cu", "gemm_tc.cu"])
def test_no_register_spills(source):
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    r = subprocess.run([nvcc, "-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-Xptxas", "-v", "-cubin", "-o", os.devnull,
                        "-I", os.path.join(b.ROOT, "include"), "-I", os.path.join(b.HERE, "csrc"), os.path.join(b.HERE, "csrc", source)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    kernels = re.findall(r"Compiling entry function '(\w+)'(?:.*\n)*?.*?(\d+) bytes spill stores, (\d+) bytes spill loads", r.stderr)
    assert kernels
    assert [k for k in kernels if k[1] != "0" or k[2] != "0"] == []


def test_no_register_spills_in_the_one_kernel_step():
    test_no_register_spills("step_cl.cu")
