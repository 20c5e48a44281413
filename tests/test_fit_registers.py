"""The error kernels hand registers from some warps to others; what their warps ask for together is what
the CTA was launched with, so the compiler has to give the kernels at least that many (96 a thread; 640
threads leave room for 102). CPU only."""

import os
import re
import subprocess

import pytest

from paper_2010_08581_gb300 import build


@pytest.mark.parametrize("src,kernel", [("fit.cu", "k_fit_tc"), ("batched_fit.cu", "kb_fit_tc")])
def test_registers_at_launch_cover_the_shares(src, kernel, tmp_path):
    text = open(os.path.join(build.CSRC, "fit_tc.cuh")).read()
    need = int(re.search(r"constexpr int FT_REGS = (\d+)", text).group(1))
    cmd = [build.nvcc(), *build.ARCH, *build.FLAGS, "-Xptxas", "-v", "-I", os.path.join(build.PKG, "..", "include"),
           "-c", os.path.join(build.CSRC, src), "-o", str(tmp_path / "x.o")]
    out = subprocess.run(cmd, capture_output=True, text=True, check=True).stderr
    entry = out[re.search(r"Compiling entry function '\S*\d" + kernel + "E", out).end():]
    assert need <= int(re.search(r"Used (\d+) registers", entry).group(1)) <= 102


@pytest.mark.parametrize("src", ["fit.cu", "batched_fit.cu"])
def test_the_library_refuses_a_kernel_with_fewer(src):
    text = open(os.path.join(build.CSRC, src)).read()
    attributes = text[text.index("fit_attributes() {"):]
    assert "fit_tc_registers(" in attributes[:attributes.index("}\n")]
