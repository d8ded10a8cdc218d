"""The float32 path where its kernels change form or run short: routes around 128 (one or two per
thread), tokens and routes that are no multiple of the staged steps (8 and 16), as many blocks of 128
tokens as take two per thread in the backward (304) and the decode (608), and one less, for the three
head sizes. Against the oracle in 64 bits.

Tolerances: the forward's products and sums are 32-bit over at most 1,000 tokens with weights that add
up to one, 1e-5 as in the parity tests; a gradient sums that many terms, 1e-5 of its own scale."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2608_11519_gb300 import flarepp, inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    flarepp.load()


SHAPES = [  # B, H, N, M, D
    (1, 1, 1, 1, 16),
    (1, 2, 17, 33, 32),
    (1, 2, 300, 127, 32),
    (2, 1, 129, 128, 16),
    (1, 1, 1000, 129, 32),
    (1, 2, 200, 130, 64),
    (19, 8, 250, 20, 16),    # 304 blocks of 128 tokens: two tokens per pair of threads
    (19, 8, 100, 9, 32),     # 152
    (19, 16, 129, 17, 32),   # 608: two tokens per thread in the decode, one in the last block
    (19, 8, 500, 8, 64),     # 608 at the head size that keeps one
]


@pytest.mark.parametrize("shape", SHAPES, ids=[str(s) for s in SHAPES])
def test_f32_kernels_match_oracle(shape):
    B, H, N, M, D = shape
    scale = 1.0 / math.sqrt(D)
    w = inputs.Workload("case", B, H, N, M, D, "f32")
    x = inputs.make_inputs(w, 31)
    dY = inputs.make_output_grad(w, 31)
    xd = {k: v.cuda() for k, v in x.items()}
    args = (xd["seeds"], xd["Kt"], xd["Vt"], xd["K"], xd["V"])
    Y, saved = flarepp.route_fwd_train(*args, scale)
    grads = flarepp.route_bwd(*args, Y, dY.cuda(), saved, scale)
    torch.cuda.synchronize()
    f = inputs.to_f64_numpy(x)
    a = (f["seeds"], f["Kt"], f["Vt"], f["K"], f["V"], scale)
    _, _, Yo = oracle.route(*a)
    err = float(np.abs(Y.double().cpu().numpy() - Yo).max())
    assert err <= 1e-5, f"Y: {err}"
    want = oracle.route_bwd(*a, dY.double().numpy())
    for name, g, r in zip(("dseeds", "dKt", "dVt", "dK", "dV"), grads, want):
        err = float(np.abs(g.double().cpu().numpy() - r).max())
        bound = 1e-5 * max(1.0, float(np.abs(r).max()))
        assert err <= bound, f"{name}: {err} > {bound}"
