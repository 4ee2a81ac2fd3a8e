"""The contraction's register shares (setmaxnreg) hold what its warps need: on tiles of up to 208 phase rows neither the
epilogue nor the control warps spill, as the compiler reports it for every instance of the kernel."""
import re
import subprocess

import pytest


def test_no_spills_on_tiles_of_208_rows(tmp_path):
    from paper_1810_06250_gb300 import builder
    try:
        nvcc = builder.nvcc()
    except RuntimeError:
        pytest.skip("nvcc not found")
    r = subprocess.run([nvcc, *builder.ARCH, *builder.FLAGS, "-Xptxas=-v", "-c", builder.CSRC + "/gemm.cu", "-o",
                        str(tmp_path / "gemm.o")], capture_output=True, text=True, check=True)
    found = re.findall(r"Compiling entry function '\S*gemm_kernelILi104E\S*'.*?(\d+) bytes spill stores, (\d+) bytes spill loads",
                       r.stderr, re.S)
    assert len(found) >= 4              # single CTAs and pairs, general and folded
    assert all(f == ("0", "0") for f in found), found
