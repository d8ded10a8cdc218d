"""Bounded waits of every tensor-core pass of the backward, each made to run out as in test_failure_gpu.py (the
load warp of CTA 0 withholds one ring item under a 1 ms limit, armed from the host): the call returns,
the status word of the backward's workspace reads the timeout, and the next backward on that workspace
matches the oracle.

Hook ids: 4 is the dZ encode where the token passes serve the shape (D <= 32, up to 512 routes at D = 32)
and the route pass of call 3 elsewhere; 8 and 9 the token pass of call 1 and that of calls 3 and 2 there,
and the separate passes of call 1 and of calls 3 and 2 together (D = 32) elsewhere; 5 to 7 the route passes
of calls 2 and 1 and the token pass of calls 3 and 2 of the separate passes."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_11519_gb300 import flarepp, inputs

pytestmark = pytest.mark.gpu

CASES = [  # hook id, N, M, D, what it withholds from
    (4, 700, 96, 32, "dZ encode"),
    (8, 700, 96, 32, "token pass of call 1 with dseeds"),
    (9, 700, 96, 32, "token pass of calls 3 and 2 with dQ"),
    (9, 700, 130, 16, "token pass of calls 3 and 2 with dQ, D = 16"),
    (4, 700, 96, 64, "route pass of call 3"),
    (5, 700, 96, 64, "route pass of call 2"),
    (6, 700, 96, 64, "route pass of call 1"),
    (7, 700, 96, 64, "token pass of calls 3 and 2"),
    (8, 700, 96, 64, "token pass of call 1"),
    (4, 300, 513, 32, "route pass of call 3, two route groups"),
    (9, 300, 513, 32, "merged token pass of calls 3 and 2"),
]


@pytest.mark.parametrize("hook,N,M,D,name", CASES, ids=[f"{c[0]}_{c[4]}" for c in CASES])
def test_wait_of_each_pass_runs_out_and_recovers(hook, N, M, D, name):
    lib = flarepp.load()
    w = inputs.Workload("timeout", 1, 2, N, M, D, "bf16")
    x = inputs.make_inputs(w, seed=23)
    dY = inputs.make_output_grad(w, 23)
    xd = {k: v.cuda() for k, v in x.items()}
    args = (xd["seeds"], xd["Kt"], xd["Vt"], xd["K"], xd["V"])
    Y, saved = flarepp.route_fwd_train(*args, w.scale)
    wsb = flarepp.Workspace()
    lib.flarepp_test_wait_fault(hook, 0, 1_000_000)
    try:
        flarepp.route_bwd(*args, Y, dY.cuda(), saved, w.scale, workspace=wsb)
        torch.cuda.synchronize()
        status = flarepp.device_status(args, wsb)
    finally:
        lib.flarepp_test_wait_fault(0, -1, 0)
    assert status == flarepp.ERR_TIMEOUT, f"{name}: status {status} after a withheld item"
    grads = flarepp.route_bwd(*args, Y, dY.cuda(), saved, w.scale, workspace=wsb)
    torch.cuda.synchronize()
    assert flarepp.device_status(args, wsb) == flarepp.OK
    f = inputs.to_f64_numpy(x)
    want = oracle.route_bwd(f["seeds"], f["Kt"], f["Vt"], f["K"], f["V"], w.scale,
                            dY.double().numpy())
    for gname, g, r in zip(("dseeds", "dKt", "dVt", "dK", "dV"), grads, want):
        bound = 2e-2 * max(1.0, float(np.abs(r).max()))
        err = float(np.abs(g.double().cpu().numpy() - r).max())
        assert err <= bound, f"after the timeout in the {name}: {gname} {err} > {bound}"
