"""Parity of the gradients where the backward's reduces share a row's partial slots out to several ways:
few routes and long sequences, rows that do not fill a block, few slots of many batch elements, and a
flagged head (its dQ is summed from the route passes' partials). Tolerances as in test_bwd_gpu.py."""
import math

import pytest
import torch

import oracle
from paper_2608_11519_gb300 import inputs
from test_bwd_gpu import TOL, _check_grads, _gpu_grads, _np, _stat_spread

pytestmark = pytest.mark.gpu

SHAPES = [  # B, H, N, M, D, dtype
    (1, 1, 20000, 16, 32, "bf16"),  # 32 ways of 420 slots
    (1, 1, 9000, 5, 16, "bf16"),    # rows end inside a block
    (1, 1, 9000, 3, 64, "bf16"),    # the separate passes
    (33, 1, 150, 9, 32, "bf16"),    # the seeds' sum over the batch
    (1, 1, 30000, 7, 16, "f32"),
    (17, 1, 200, 4, 64, "f32"),
    (2, 1, 500, 150, 64, "f32"),    # two threads per route in call 3, a ragged route tile
    (38, 8, 249, 9, 32, "f32"),     # two tokens per pair of threads, 608 blocks of them
    (57, 8, 113, 7, 16, "f32"),     # and 456
]


@pytest.mark.parametrize("shape", SHAPES, ids=[str(s) for s in SHAPES])
def test_shared_slots_match_oracle(shape):
    B, H, N, M, D, dt = shape
    w = inputs.Workload("case", B, H, N, M, D, dt)
    x = inputs.make_inputs(w, 31)
    dY = inputs.make_output_grad(w, 31)
    s = 1.0 / math.sqrt(D)
    got, _ = _gpu_grads(x, dY, s)
    f = inputs.to_f64_numpy(x)
    want = oracle.route_bwd(f["seeds"], f["Kt"], f["Vt"], f["K"], f["V"], s, _np(dY))
    _check_grads(got, want, TOL[dt])


def test_flagged_head_with_few_routes():
    w = inputs.Workload("case", 1, 2, 9000, 20, 32, "bf16")
    s = 1.0 / math.sqrt(w.D)
    x = inputs.make_inputs(w, 5)
    x["seeds"] = (x["seeds"].float() * 10).to(torch.bfloat16)
    K = x["K"].float()
    K[:, 1] *= 16
    x["K"] = K.to(torch.bfloat16)
    dY = inputs.make_output_grad(w, 5)
    f = inputs.to_f64_numpy(x)
    spread = _stat_spread(f, s)
    assert spread[0] < 60.0 < spread[1], spread
    got, _ = _gpu_grads(x, dY, s)
    want = oracle.route_bwd(f["seeds"], f["Kt"], f["Vt"], f["K"], f["V"], s, _np(dY))
    _check_grads(got, want, TOL["bf16"])
