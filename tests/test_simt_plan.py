"""The float32 passes' chunk plans (make_plan and make_bwd_plan, plan.cu, compiled here as host code): the
waves of CTAs take little more than an even share of the tokens, whatever the batch and the width of the
route tiles, without more chunks than the merge can take, and more chunks never take a shape from the call that works in a fixed scratch of 64 MiB
(the plan that this is held against cut the tokens for about four waves of CTAs)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2608_11519_gb300", "csrc")

HARNESS = r"""
#include <math.h>
#include <stdio.h>
#include <random>
#include "flarepp_internal.h"
using namespace flarepp;

namespace flarepp {  // (of the tensor-core path, which is not planned here)
int64_t tc_encode_item_rows(int64_t) { return 96; }
int64_t tc_group_rows(int64_t) { return 512; }
}  // namespace flarepp

static int64_t up(int64_t x) { return (x + 255) / 256 * 256; }

int main() {
    int bad = 0, n = 0, scratch = 0;
    // warps that a quarter of an SM's 64K registers holds, four times
    auto warps = [](int regs) { return 4 * (16384 / ((regs + 7) / 8 * 8 * 32)); };
    auto check = [&](int64_t B, int64_t H, int64_t N, int64_t M, int64_t D) {
        flarepp_shape s{B, H, N, M, D, FLAREPP_F32};
        Plan p;
        if (make_plan(&s, &p) != FLAREPP_OK) return;
        const BwdPlan b = make_bwd_plan(p);
        const int64_t bh = B * H, tile = M >= 128 ? 128 : cdiv(M, 32) * 32, tiles = bh * cdiv(M, tile);
        const bool two = M >= 128 && D <= 32;
        const int64_t enc = warps(two ? 168 : (D == 16 ? 168 : 255)) / (two ? 2 : tile / 32);
        const int64_t route = warps(D == 16 ? 128 : 255) / (tile / 32);
        // the waves' tokens and the merge's chunks (in tokens: 0.04 us each in the encode's) beside an
        // even share and what balancing the two has to leave
        auto fits = [&](int64_t len, int64_t chunks, int64_t places, double bytes, double cap,
                        double merge) {
            const double time = (double)cdiv(tiles * chunks, places * kNumSMs) * (double)len;
            const double share = (double)tiles * (double)N / (double)(places * kNumSMs);
            const double even = sqrt((merge + bytes / 0.56e6) * (double)N);
            return len % 16 == 0 && chunks == cdiv(N, len) &&
                   (time + merge * (double)chunks <=
                        1.6 * share + 64.0 + 2.5 * even + 16.0 * (double)cdiv(tiles, places * kNumSMs) ||
                    4.0 * (double)chunks * bytes > cap);  // (or more partials would take too much)
        };
        const double e = (double)bh * M * (D + 2) * 4.0;
        const bool ok = fits(p.chunk_len, p.nchunk, enc, e, 32e6, D == 16 ? 1.0 : (D == 32 ? 0.4 : 0.15)) &&
                        fits(b.chunk_len, b.nchunk, route, (double)bh * M * D * 4.0, 32e6, 0.03) &&
                        (p.nchunk == 1 || (double)p.nchunk * e <= 32.0 * 1048576.0);
        // the workspace with chunks for four waves of 608 CTAs
        int64_t want = cdiv(608, tiles);
        const int64_t rows = bh * cdiv(N, cdiv(cdiv(N, want), 32) * 32) * M;
        const int64_t before = 256 + 2 * up(rows * 4) + up(rows * D * 4) + 2 * up(bh * M * D * 4);
        const bool taken = before > (64 << 20) || p.total <= (64u << 20);
        scratch += before <= (64 << 20);
        ++n;
        if ((!ok || !taken) && bad++ < 8)
            printf("B=%ld H=%ld N=%ld M=%ld D=%ld: %ld x %ld, %ld x %ld, %zu bytes (%ld)\n", (long)B,
                   (long)H, (long)N, (long)M, (long)D, (long)p.nchunk, (long)p.chunk_len,
                   (long)b.nchunk, (long)b.chunk_len, p.total, (long)before);
    };
    for (int64_t B : {1, 2, 20, 32, 40})
        for (int64_t H : {1, 5, 8})
            for (int64_t N : {1, 15, 781, 1024, 16384, 20000, 60000, 262144})
                for (int64_t M : {1, 16, 32, 33, 64, 96, 100, 128, 256, 300, 2048})
                    for (int64_t D : {16, 32, 64}) check(B, H, N, M, D);
    std::mt19937_64 g(9);
    for (int i = 0; i < 20000; ++i)
        check(1 + g() % 64, 1 + g() % 16, 1 + g() % (g() % 2 ? 3000 : 300000), 1 + g() % 2048,
              16 << (g() % 3));
    printf("%d shapes (%d within the scratch before), %d wrong\n", n, scratch, bad);
    return bad != 0;
}
"""


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="nvcc not found")
def test_float32_chunks_fill_the_machine_within_the_scratch(tmp_path):
    src = tmp_path / "plan.cu"
    src.write_text(HARNESS)
    exe = tmp_path / "plan"
    subprocess.run(["nvcc", "-std=c++17", "-O2", "-I", CSRC, "-I", os.path.join(ROOT, "include"),
                    str(src), os.path.join(CSRC, "plan.cu"), "-o", str(exe)], check=True,
                   capture_output=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
