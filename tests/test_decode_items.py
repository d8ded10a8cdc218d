"""The width of the decode's items (tc_decode_item_rows, tc_kernels.cu, called here on the host): as few
items per unit as its forms allow, and among forms with as many the narrower one, whose columns beyond
the last route are fewer (at D = 64, 144 routes are three items of 48 or of 64)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2608_11519_gb300", "csrc")

HARNESS = r"""
#include <stdio.h>
#include "flarepp_internal.h"

namespace flarepp {
cudaError_t ensure_smem_limit(const void*, int) { return cudaErrorInvalidValue; }
}  // namespace flarepp

int main() {
    for (int D = 16; D <= 64; D *= 2)
        for (int M = 1; M <= 2048; ++M)
            printf("%d %d %d %d\n", D, M, (int)flarepp::tc_decode_item_rows(D, M, false),
                   D <= 32 ? (int)flarepp::tc_decode_item_rows(D, M, true) : 0);
    return 0;
}
"""

FORMS = {16: (64, 112), 32: (64, 96), 64: (48, 64)}


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="nvcc not found")
def test_decode_items_are_few_and_then_narrow(tmp_path):
    src = tmp_path / "items.cu"
    src.write_text(HARNESS)
    exe = tmp_path / "items"
    subprocess.run(["nvcc", "-std=c++17", "-O0", "--expt-relaxed-constexpr", "-gencode",
                    "arch=compute_103a,code=sm_103a", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                    str(src), os.path.join(CSRC, "tc_kernels.cu"), "-o", str(exe)], check=True,
                   capture_output=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120, check=True).stdout
    rows = [tuple(int(v) for v in line.split()) for line in out.splitlines()]
    assert len(rows) == 3 * 2048
    for D, M, rows_per_item, lo in rows:
        narrow, wide = FORMS[D]
        want = wide if -(-M // wide) < -(-M // narrow) else narrow
        assert rows_per_item == want, (D, M)
        if D <= 32:
            assert lo == narrow, (D, M)
