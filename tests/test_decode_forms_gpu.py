"""GPU parity of the decode's two forms (64-route items, and items as wide as TMEM allows) at the
route counts around an item's edge, where the form changes and where the last item holds one route
or a chunk without any. Tolerance as in test_parity_gpu.py (bf16: 2e-2)."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2608_11519_gb300 import flarepp, inputs

pytestmark = pytest.mark.gpu

CASES = [(32, m) for m in (64, 65, 96, 97, 128, 129, 192, 193, 225, 289)] + \
        [(16, m) for m in (64, 65, 112, 113, 128, 129, 225, 241)] + \
        [(64, m) for m in (1, 63, 64, 65, 129)]


@pytest.mark.parametrize("D,M", CASES)
def test_decode_matches_oracle(D, M):
    w = inputs.Workload("case", 2, 2, 1100, M, D, "bf16")
    x = inputs.make_inputs(w, 8)
    xd = {k: v.cuda() for k, v in x.items()}
    Y = flarepp.route_fwd(xd["seeds"], xd["Kt"], xd["Vt"], xd["K"], xd["V"])
    F = flarepp.flare_fwd(xd["seeds"], xd["K"], xd["V"])
    torch.cuda.synchronize()
    f = inputs.to_f64_numpy(x)
    s = 1.0 / math.sqrt(D)
    want = oracle.route(f["seeds"], f["Kt"], f["Vt"], f["K"], f["V"], s)[2]
    assert float(np.abs(Y.double().cpu().numpy() - want).max()) <= 2e-2
    q = np.broadcast_to(f["seeds"], (w.B,) + f["seeds"].shape)
    z, _ = oracle.sdpa(q, f["K"], f["V"], s)
    want, _ = oracle.sdpa(f["K"], q, z, s)
    assert float(np.abs(F.double().cpu().numpy() - want).max()) <= 2e-2
