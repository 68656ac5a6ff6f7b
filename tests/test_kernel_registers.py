"""The tensor-core kernel's epilogue with a residual and per-channel integer constants fills the 96 registers of two CTAs an SM:
what the compiler spills there costs every tile (128 bytes of it: 4 to 19 % of a layer)."""
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1805_07941_b200", "csrc")

SOURCE = """
#include <algorithm>
#include <vector>
#include "epilogue.cuh"
#include "kernel_igemm.cuh"
namespace qc {
decltype(&igemm_i8_kernel<EPI_FAST_I8_RES>) kernel = igemm_i8_kernel<EPI_FAST_I8_RES>;
}
"""


def test_the_integer_residual_epilogue_spills_little(tmp_path):
    source = tmp_path / "kernel.cu"
    source.write_text(SOURCE)
    out = subprocess.run(["nvcc", "-gencode", "arch=compute_100a,code=sm_100a", "-O3", "-std=c++17", "-Xptxas", "-v", "-I", CSRC, "-c",
                          "-o", str(tmp_path / "kernel.o"), str(source)], capture_output=True, text=True, check=True, timeout=300).stderr
    entry = out[re.search(r"Compiling entry function '\S*igemm_i8_kernel", out).start():]
    assert int(re.search(r"(\d+) bytes spill stores", entry).group(1)) <= 76, entry[:400]
    assert int(re.search(r"Used (\d+) registers", entry).group(1)) <= 96
