"""How the backward's reduces share out a row's partial slots (reduce_ways, compiled here as host code): no
way is left with a long chain of loads while the machine has room, and the ways divide a block into
whole rows."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2608_11519_gb300", "csrc")

HARNESS = r"""
#include <stdio.h>
#include "flarepp_internal.h"
using namespace flarepp;

int main() {
    int bad = 0, n = 0;
    for (int64_t D : {16, 32, 64})
        for (int64_t rows = 1; rows <= 600000; rows += 1 + rows / 3)
            for (int64_t slots = 1; slots <= 3000; slots += 1 + slots / 4) {
                const int64_t ways = reduce_ways(rows, D, slots), most = D == 64 ? 16 : 32;
                const bool shape = ways >= 1 && ways <= most && (ways & (ways - 1)) == 0 &&
                                   (kRedThreads / ways) % (D / 4) == 0;
                const bool shared = ways == most || slots <= 8 * ways ||
                                    rows * (D / 4) * ways >= 2 * kRedThreads * kNumSMs;
                const bool idle = ways > 1 && slots <= 4 * ways;  // ways beyond what the slots ask for
                ++n;
                if ((!shape || !shared || idle) && bad++ < 5)
                    printf("D=%d rows=%d slots=%d: %d\n", (int)D, (int)rows, (int)slots, (int)ways);
            }
    printf("%d shapes, %d wrong\n", n, bad);
    return bad != 0;
}
"""


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="nvcc not found")
def test_ways_leave_no_long_chain(tmp_path):
    src = tmp_path / "ways.cu"
    src.write_text(HARNESS)
    exe = tmp_path / "ways"
    subprocess.run(["nvcc", "-std=c++17", "-O2", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                    str(src), "-o", str(exe)], check=True, capture_output=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
