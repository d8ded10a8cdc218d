"""The float32 kernels keep their rows and sums in registers: no kernel of simt_f32.cu or of the backward's
CUDA-core passes (bwd.cu) spills more than 160 bytes per thread, by the assembler's report."""
import os
import re
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2608_11519_gb300", "csrc")


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="nvcc not found")
@pytest.mark.parametrize("unit", ["simt_f32.cu", "bwd.cu"])
def test_float32_kernels_stay_in_registers(tmp_path, unit):
    r = subprocess.run(["nvcc", "-gencode", "arch=compute_103a,code=sm_103a", "-O3", "-std=c++17",
                        "--expt-relaxed-constexpr", "-I", os.path.join(ROOT, "include"), "-Xptxas", "-v",
                        "-c", os.path.join(CSRC, unit), "-o", str(tmp_path / "unit.o")],
                       capture_output=True, text=True, check=True)
    spills = {}
    for part in (r.stdout + r.stderr).split("Compiling entry function")[1:]:
        name = re.search(r"(simt_encode|simt_decode|route_pass|token_pass)_kernelI(\w*?)EEE?v", part)
        if name:
            spills[name.group(0)] = int(re.search(r"(\d+) bytes spill stores", part).group(1))
    assert len(spills) >= 10
    assert max(spills.values()) <= 160, spills
