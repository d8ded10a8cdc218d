"""The mixer's projections and weight gradients where their tiles change form: row tiles taken in
pairs (from 304 tiles of 128 tokens on, in the products that read the heads' tensors), an odd number
of them, a last one of a few rows, pairs that would cross from one batch element into the next; column
tiles that span two projections; and the weight gradients' items of 256 rows, whole and cut short.
Layer and gradients against the oracle, each within 2e-2 of its own scale as in the parity tests (bf16
operands and results, float32 sums)."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2608_11519_gb300 import flarepp

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    flarepp.load()


SHAPES = [  # B, H, N, M, D, P
    (1, 2, 303 * 128, 16, 32, 4),      # 303 row tiles: one at a time
    (1, 2, 303 * 128 + 5, 16, 32, 2),  # 304: pairs, five rows in the last tile
    (1, 1, 304 * 128 + 1, 16, 16, 4),  # 305: the last pair has one tile, of one row
    (102, 1, 300, 16, 64, 2),          # three row tiles per batch element: a pair and a single
    (3, 3, 200, 16, 32, 4),            # four heads per column tile of twelve, three per projection
    (160, 1, 70, 16, 32, 2),           # more weight-gradient items than SMs, six tokens in a last stage
    (2, 5, 130, 16, 64, 4),            # C = 320: weight-gradient rows in 128s, the last half of an item
]


def _np(t):
    return t.detach().to("cpu", torch.float64).numpy()


@pytest.mark.parametrize("shape", SHAPES, ids=[str(s) for s in SHAPES])
def test_projection_tiles_match_oracle(shape):
    B, H, N, M, D, P = shape
    C = H * D
    g = torch.Generator().manual_seed(5)
    X = torch.randn(B, N, C, generator=g).to(torch.bfloat16)
    W_in = (torch.randn(P * C, C, generator=g) / math.sqrt(C)).to(torch.bfloat16)
    Wo = (torch.randn(C, C, generator=g) / math.sqrt(C)).to(torch.bfloat16)
    seeds = torch.randn(H, M, D, generator=g).to(torch.bfloat16)
    dO = torch.randn(X.shape, generator=g).to(torch.bfloat16)
    s = 1.0 / math.sqrt(D)
    dev = [t.cuda() for t in (X, W_in, Wo, seeds)]
    O, saved = flarepp.mixer_fwd_train(*dev, s)
    grads = flarepp.mixer_bwd(*dev, saved, dO.cuda(), s)
    torch.cuda.synchronize()
    f = [_np(t) for t in (X, W_in, Wo, seeds)]
    want = (oracle.mixer(*f, s),) + tuple(oracle.mixer_bwd(*f, s, _np(dO)))
    for name, got, ref in zip(("O", "dX", "dW_in", "dWo", "dseeds"), (O,) + tuple(grads), want):
        bound = 2e-2 * max(1.0, float(np.abs(ref).max()))
        err = float(np.abs(_np(got) - ref).max())
        assert err <= bound, f"{name}: {err} > {bound}"
