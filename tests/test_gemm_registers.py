"""What ptxas reports for the GEMM kernels: no thread keeps anything in local memory."""
import os
import re
import subprocess

from paper_2507_14959_b200 import build


def test_no_gemm_kernel_spills(tmp_path):
    log = subprocess.run([build.nvcc_path(), "-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-I", os.path.join(build.ROOT, "include"),
                          "-I", build.CSRC, "-Xptxas", "-v", "-cubin", os.path.join(build.CSRC, "gemm_tcgen05.cu"), "-o", str(tmp_path / "gemm.cubin")],
                         capture_output=True, text=True, check=True).stderr
    used = re.findall(r"Function properties for (\S*lora_gemm\S*)\s+(\d+) bytes stack frame, (\d+) bytes spill stores", log)
    assert len(used) >= 20
    assert [u for u in used if (u[1], u[2]) != ("0", "0")] == []
