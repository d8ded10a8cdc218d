"""GPU parity of the token passes that also form dQ (tc_tok.cu) at the sizes where they can go
wrong: one item, one stream without an item, ragged route items and token tiles, several (b, h)
in one CTA's run of tiles, the largest route counts they serve and one more (which the separate
passes take). Tolerance as in test_bwd_gpu.py: 2e-2 of each gradient's scale."""
import math

import numpy as np
import pytest
import torch

import oracle
from paper_2608_11519_gb300 import flarepp, inputs

pytestmark = pytest.mark.gpu

SHAPES = [
    # B, H, N, M, D, scale (None: 1/sqrt(D))
    (1, 1, 1, 1, 32, None),        # one token, one route
    (1, 2, 129, 64, 32, None),     # one item: the second stream idles; a second tile of one token
    (2, 1, 128, 65, 16, None),     # the second item has one route
    (1, 3, 300, 127, 32, None),
    (1, 1, 257, 129, 16, None),    # a second block of one route, no item in its second half
    (3, 5, 1500, 192, 32, None),   # 180 tiles: CTAs with two tiles and two (b, h)
    (40, 8, 100, 40, 16, None),    # 320 (b, h) of one tile each: three segments per CTA
    (1, 2, 400, 512, 32, -0.2),    # the largest M at D = 32; negative scale
    (1, 1, 200, 513, 32, None),    # beyond it: the separate passes
    (1, 1, 300, 1024, 16, None),   # the largest M at D = 16
    (1, 1, 200, 1025, 16, None),
]


@pytest.mark.parametrize("shape", SHAPES, ids=[str(s) for s in SHAPES])
def test_token_passes_match_oracle(shape):
    B, H, N, M, D, scale = shape
    scale = 1.0 / math.sqrt(D) if scale is None else scale
    w = inputs.Workload("case", B, H, N, M, D, "bf16")
    x = inputs.make_inputs(w, 12)
    dY = inputs.make_output_grad(w, 12)
    xd = {k: v.cuda() for k, v in x.items()}
    args = (xd["seeds"], xd["Kt"], xd["Vt"], xd["K"], xd["V"])
    ws = flarepp.Workspace()
    Y, saved = flarepp.route_fwd_train(*args, scale)
    grads = flarepp.route_bwd(*args, Y, dY.cuda(), saved, scale, workspace=ws)
    torch.cuda.synchronize()
    assert flarepp.device_status(args, ws) == flarepp.OK
    f = inputs.to_f64_numpy(x)
    want = oracle.route_bwd(f["seeds"], f["Kt"], f["Vt"], f["K"], f["V"], scale,
                            dY.double().numpy())
    for name, g, r in zip(("dseeds", "dKt", "dVt", "dK", "dV"), grads, want):
        err = float(np.abs(g.double().cpu().numpy() - r).max())
        bound = 2e-2 * max(1.0, float(np.abs(r).max()))
        assert err <= bound, f"{name}: {err} > {bound}"


@pytest.mark.parametrize("N,M,D", [(4097, 130, 32)])
def test_flagged_heads_over_several_slices(N, M, D):
    """The ranges of the log-normalisers are taken over slices of 4,096 tokens; one token more makes
    two. Keys x 16 on head 1 take it out of the merged pass's range while head 0 stays; both match
    the oracle at the bf16 tolerance."""
    from test_bwd_gpu import _stat_spread
    scale = 1.0 / math.sqrt(D)
    w = inputs.Workload("case", 1, 2, N, M, D, "bf16")
    x = inputs.make_inputs(w, 5)
    x["seeds"] = (x["seeds"].float() * 10).to(torch.bfloat16)
    K = x["K"].float()
    K[:, 1] *= 16
    x["K"] = K.to(torch.bfloat16)
    dY = inputs.make_output_grad(w, 5)
    f = inputs.to_f64_numpy(x)
    spread = _stat_spread(f, scale)
    assert spread[0] < 60.0 < spread[1], spread
    xd = {k: v.cuda() for k, v in x.items()}
    args = (xd["seeds"], xd["Kt"], xd["Vt"], xd["K"], xd["V"])
    Y, saved = flarepp.route_fwd_train(*args, scale)
    grads = flarepp.route_bwd(*args, Y, dY.cuda(), saved, scale)
    torch.cuda.synchronize()
    want = oracle.route_bwd(f["seeds"], f["Kt"], f["Vt"], f["K"], f["V"], scale,
                            dY.double().numpy())
    for name, g, r in zip(("dseeds", "dKt", "dVt", "dK", "dV"), grads, want):
        err = float(np.abs(g.double().cpu().numpy() - r).max())
        bound = 2e-2 * max(1.0, float(np.abs(r).max()))
        assert err <= bound, f"{name}: {err} > {bound}"
