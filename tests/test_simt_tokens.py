"""When the float32 backward's token passes take two tokens per pair of threads (simt_two_tokens, compiled
here as host code): where their blocks fill whole waves, and not where a few blocks would open one more
wave, nor where the machine is far from full. Both forms are measured at these sizes."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2608_11519_gb300", "csrc")

# D, call 1, N, BH: two tokens are faster
CASES = [
    (32, 0, 16384, 8, 1), (32, 1, 16384, 8, 1), (16, 0, 16384, 8, 1), (16, 1, 16384, 8, 1),
    (16, 1, 60000, 8, 1),
    (32, 0, 249, 304, 1), (32, 1, 249, 304, 1), (16, 0, 113, 456, 1), (16, 1, 113, 456, 1),
    (16, 0, 60000, 1, 0), (16, 1, 60000, 1, 0),  # 469 blocks of 128 tokens, 456 places
    (16, 1, 781, 160, 0),
    (32, 0, 1024, 4, 0), (32, 1, 1024, 4, 0), (16, 0, 500, 1, 0),
    (64, 0, 16384, 8, 0), (64, 1, 16384, 8, 0),
]


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="nvcc not found")
def test_two_tokens_only_where_they_are_faster(tmp_path):
    calls = "\n".join(f'    printf("%d\\n", (int)flarepp::simt_two_tokens({d}, {c}, {n}, {bh}));'
                      for d, c, n, bh, _ in CASES)
    src = tmp_path / "two.cu"
    src.write_text('#include <stdio.h>\n#include "flarepp_internal.h"\nint main() {\n' + calls + "\n}\n")
    exe = tmp_path / "two"
    subprocess.run(["nvcc", "-std=c++17", "-I", CSRC, "-I", os.path.join(ROOT, "include"), str(src),
                    "-o", str(exe)], check=True, capture_output=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()
    assert [int(v) for v in out] == [c[-1] for c in CASES]
