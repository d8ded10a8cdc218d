"""The input projection (tc_gemm.cu) with one, two and four output tensors reads exactly as many output
pointers as it is given: its host code, compiled with AddressSanitizer, runs on a heap array of P
pointers. No GPU is used: without a driver the call ends when it asks for the tensor maps, after it has
read the pointers."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2608_11519_gb300", "csrc")

HARNESS = r"""
#include <stdio.h>
#include <stdlib.h>
#include "flarepp_internal.h"

namespace flarepp {
cudaError_t ensure_smem_limit(const void*, int) { return cudaErrorInvalidValue; }
}  // namespace flarepp

int main(int argc, char** argv) {
    const int P = atoi(argv[1]);
    alignas(16) static char tensor[4096];
    void** outs = new void*[P];
    for (int p = 0; p < P; ++p) outs[p] = tensor;
    const cudaError_t e = flarepp::tc_projection(1, 4, 2, 16, P, tensor, tensor, outs, nullptr, 0);
    delete[] outs;
    printf("ended with %d\n", (int)e);
    return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    if shutil.which("nvcc") is None:
        pytest.skip("nvcc not found")
    tmp = tmp_path_factory.mktemp("projection")
    src = tmp / "outputs.cu"
    src.write_text(HARNESS)
    exe = tmp / "outputs"
    subprocess.run(["nvcc", "-std=c++17", "-O1", "--expt-relaxed-constexpr", "-gencode",
                    "arch=compute_103a,code=sm_103a", "-Xcompiler", "-fsanitize=address",
                    "-I", CSRC, "-I", os.path.join(ROOT, "include"), str(src),
                    os.path.join(CSRC, "tc_gemm.cu"), "-o", str(exe)], check=True,
                   capture_output=True)
    return str(exe)


@pytest.mark.parametrize("P", [1, 2, 4])
def test_projection_reads_only_its_output_pointers(program, P):
    env = dict(os.environ, CUDA_VISIBLE_DEVICES="", ASAN_OPTIONS="detect_leaks=0:protect_shadow_gap=0")
    r = subprocess.run([program, str(P)], capture_output=True, text=True, timeout=120, env=env)
    assert r.returncode == 0 and "ended with" in r.stdout, r.stdout + r.stderr
