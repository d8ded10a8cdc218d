"""Heads whose log-normalisers spread too far for the merged passes (flagged heads), where skipping them can
go wrong: between served heads inside one CTA's run of token tiles (first, middle and last heads of a
run, several in a row), and in the separate passes of more routes than the token passes take (the merged
pass serves some heads and the unmerged one the rest). Every gradient at the bf16 tolerance of
test_bwd_gpu.py (an emulation of the passes in float64 with their roundings takes at most 0.7 of it on
these inputs; of a few short, sharper heads it takes more)."""
import math

import pytest
import torch

import oracle
from paper_2608_11519_gb300 import inputs
from test_bwd_gpu import TOL, _check_grads, _gpu_grads, _np, _stat_spread

pytestmark = pytest.mark.gpu

CASES = [  # B, H, N, M, D, heads whose keys are scaled by 16, scale of the seeds
    (40, 8, 130, 20, 32, (0, 3, 4, 7), 10),  # 640 tiles: runs of four or five, two tiles a (b, h)
    (50, 8, 100, 40, 16, (2, 5), 4),         # 400 tiles: two or three (b, h) a run
    (76, 2, 300, 33, 32, (1,), 10),          # 456 tiles of three a (b, h): every run one (b, h)
    (1, 4, 700, 530, 32, (1, 3), 10),        # beyond the token passes' routes
]


@pytest.mark.parametrize("B,H,N,M,D,heads,sharp", CASES, ids=[str(c) for c in CASES])
def test_flagged_heads_match_oracle(B, H, N, M, D, heads, sharp):
    scale = 1.0 / math.sqrt(D)
    w = inputs.Workload("case", B, H, N, M, D, "bf16")
    x = inputs.make_inputs(w, 5)
    x["seeds"] = (x["seeds"].float() * sharp).to(torch.bfloat16)
    K = x["K"].float()
    for h in heads:
        K[:, h] *= 16
    x["K"] = K.to(torch.bfloat16)
    dY = inputs.make_output_grad(w, 5)
    f = inputs.to_f64_numpy(x)
    spread = _stat_spread(f, scale)
    wide = [s > 60.0 for s in spread]
    for h in range(H):
        of_head = [wide[b * H + h] for b in range(B)]
        assert any(of_head) == (h in heads), (h, spread[h::H])
    got, _ = _gpu_grads(x, dY, scale)
    want = oracle.route_bwd(f["seeds"], f["Kt"], f["Vt"], f["K"], f["V"], scale, _np(dY))
    _check_grads(got, want, TOL["bf16"])
