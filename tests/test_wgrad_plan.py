"""The weight gradients' plan (wgrad_plan, tc_wgrad.cu, called here on the host) keeps the SMs busy: the
time of its waves, in stages of 64 tokens, stays near an even share of all stages, whatever the batch,
and the partial sums fit the bytes it asks for."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2608_11519_gb300", "csrc")

HARNESS = r"""
#include <stdio.h>
#include <random>
#include "flarepp_internal.h"
using namespace flarepp;

namespace flarepp {
cudaError_t ensure_smem_limit(const void*, int) { return cudaErrorInvalidValue; }
}  // namespace flarepp

int main() {
    int bad = 0, n = 0;
    auto check = [&](int64_t B, int64_t N, int64_t R, int64_t C) {
        const WgradPlan w = wgrad_plan(B, N, R, C);
        const int64_t stages = B * cdiv(N, 64), tiles = w.row_groups * w.col_tiles;
        const int64_t waves = cdiv(tiles * w.n_chunks, kNumSMs);
        const double time = (double)waves * (double)cdiv(stages, w.n_chunks);
        const double share = (double)tiles * (double)stages / kNumSMs;
        const bool ok = w.n_chunks >= 1 && w.n_chunks <= stages && time <= 1.35 * share + 16.0 &&
                        w.part_bytes == (size_t)w.n_chunks * R * C * 4;
        ++n;
        if (!ok && bad++ < 8)
            printf("B=%ld N=%ld R=%ld C=%ld: %ld chunks, %g stages, an even share is %g\n", (long)B,
                   (long)N, (long)R, (long)C, (long)w.n_chunks, time, share);
    };
    for (int64_t B : {1, 2, 3, 10, 13, 20, 32, 40, 100, 160})
        for (int64_t N : {1, 64, 1000, 2000, 16384, 262144})
            for (int64_t C : {16, 32, 96, 128, 256, 320, 512, 1024, 2048})
                for (int64_t p : {1, 4}) check(B, N, p * C, C);
    std::mt19937_64 g(3);
    for (int i = 0; i < 5000; ++i) {
        const int64_t C = 16 * (1 + g() % 64);
        check(1 + g() % 64, 1 + g() % 100000, (g() % 2 ? 4 : 1) * C, C);
    }
    printf("%d shapes, %d wrong\n", n, bad);
    return bad != 0;
}
"""


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="nvcc not found")
def test_weight_gradient_items_fill_the_machine(tmp_path):
    src = tmp_path / "plan.cu"
    src.write_text(HARNESS)
    exe = tmp_path / "plan"
    subprocess.run(["nvcc", "-std=c++17", "-O1", "--expt-relaxed-constexpr", "-gencode",
                    "arch=compute_103a,code=sm_103a", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                    str(src), os.path.join(CSRC, "tc_wgrad.cu"), "-o", str(exe)], check=True,
                   capture_output=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
