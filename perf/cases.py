"""The calls by which this library's speed is judged: the public entry points of
``paper_2608_11519_gb300.flarepp`` at the shapes that its workloads, tests and benchmark use.

A case is a dict of plain values: ``op`` (which entry point), ``dtype``, the shape B, H, N, M, D,
``centres`` (0: i.i.d. keys; else the keys of each head sit around that many centres, as tokens
of a smooth field do), ``n_proj`` (the mixer's projections) and ``scale`` (None: 1/sqrt(D)).

    chain        route_fwd                    Y
    flare        flare_fwd                    Y
    train        route_fwd_train, route_bwd   Y, dseeds, dKt, dVt, dK, dV
    mixer        mixer_fwd                    O
    mixer_train  mixer_fwd_train, mixer_bwd   O, dX, dW_in, dWo, dseeds

A program keeps the workspace between calls (``flarepp.Workspace``); outputs are new tensors of
each call.
"""
import math

import torch

from paper_2608_11519_gb300 import flarepp

_TORCH = {"f32": torch.float32, "bf16": torch.bfloat16}


def _case(name, op, dtype, B, H, N, M, D, centres=0, n_proj=0, scale=None):
    c = {"op": op, "dtype": dtype, "B": B, "H": H, "N": N, "M": M, "D": D, "centres": centres,
         "n_proj": n_proj, "scale": scale}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest call: the parity workload, float32 (the paper trains in FP32)
        _case("tiny_f32", "chain", "f32", 1, 4, 1024, 32, 16),
        # a float32 training step on a 2D mesh of 16K points
        _case("pde2d_f32_train", "train", "f32", 1, 8, 16384, 128, 32, centres=64),
        # inference on a batch of 2D meshes of 16K points, peaked softmaxes
        _case("pde2d", "chain", "bf16", 4, 8, 16384, 128, 32, centres=64),
        # long-sequence classification: many short sequences
        _case("longseq", "chain", "bf16", 32, 8, 4096, 256, 32),
        # inference on a 3D mesh of a million points: the headline workload
        _case("mesh3d", "chain", "bf16", 1, 8, 1048576, 512, 32, centres=4096),
        # few routes and narrow heads on a long sequence: the memory-bound corner of the sweep
        _case("few_routes_D16", "chain", "bf16", 1, 8, 262144, 64, 16),
        # wide heads at sizes that are no multiple of any tile
        _case("ragged_D64", "chain", "bf16", 3, 5, 20011, 300, 64, centres=64),
        # FLARE (fixed learned queries) on the long-sequence shape
        _case("longseq_flare", "flare", "bf16", 32, 8, 4096, 256, 32),
        # one training step of the chain on the batch of 2D meshes
        _case("pde2d_train", "train", "bf16", 4, 8, 16384, 128, 32, centres=64),
        # one training step of the chain on a 3D mesh of 262,144 points
        _case("mesh_train", "train", "bf16", 1, 8, 262144, 512, 32, centres=1024),
        # inference of a whole mixer layer on the batch of 2D meshes
        _case("pde2d_mixer", "mixer", "bf16", 4, 8, 16384, 128, 32, n_proj=4),
        # one training step of a whole mixer layer on 262,144 points
        _case("mesh_mixer_train", "mixer_train", "bf16", 1, 8, 262144, 512, 32, n_proj=4),
    ]


# (b, h, token, route) quadruples a drawn case may have, by op and dtype, counting at least 128
# routes (256 in a training step): such a case costs no more than the largest listed one
_MOST = {("chain", "bf16"): 2.0e9, ("flare", "bf16"): 2.0e9, ("train", "bf16"): 5.0e8,
         ("mixer", "bf16"): 1.0e9, ("mixer_train", "bf16"): 5.0e8, ("chain", "f32"): 5.0e7,
         ("flare", "f32"): 5.0e7, ("train", "f32"): 1.6e7}


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["chain", "chain", "chain", "flare", "train", "train", "mixer", "mixer_train"])
    dtype = "bf16" if op.startswith("mixer") or rng.random() < 0.75 else "f32"
    while True:
        B, D = _log(rng, 1, 32), rng.choice([16, 32, 32, 64])
        H = rng.choice([2, 4, 8] if op.startswith("mixer") else [1, 2, 4, 5, 8])
        N, M = _log(rng, 500, 600000), _log(rng, 16, 2048)
        if rng.random() < 0.3:
            M = 1 << (M.bit_length() - 1)
        # not above the op's most, the inputs within a few GB, and no call smaller than any of
        # the workloads'
        cost = B * H * N * max(M, 256 if "train" in op else 128)
        if dtype == "f32":
            cost = B * H * N * max(M, 32)
        if B * H * N * M >= 1.0e5 and cost <= _MOST[op, dtype] and B * H * N * D <= 3.0e8:
            break
    n_proj = rng.choice([2, 4]) if op.startswith("mixer") else 0
    centres = 0 if n_proj or rng.random() < 0.5 else rng.choice([64, 256, 1024])
    scale = round(rng.uniform(0.05, 0.3), 3) if rng.random() < 0.2 else None
    return _case(None, op, dtype, B, H, N, M, D, centres, n_proj, scale)


def _scale(c):
    return 1.0 / math.sqrt(c["D"]) if c["scale"] is None else c["scale"]


def _inputs(c, seed):
    """The input tensors, on the GPU, from the seed alone."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    B, H, N, M, D, dt = c["B"], c["H"], c["N"], c["M"], c["D"], _TORCH[c["dtype"]]

    def normal(*shape, std=1.0):
        return (torch.randn(*shape, generator=g, device="cuda") * std).to(dt)

    def keys():
        if not c["centres"]:
            return normal(B, H, N, D)
        centre = torch.randn(H * c["centres"], D, generator=g, device="cuda") * 1.5
        pick = torch.randint(0, c["centres"], (B, H, N), generator=g, device="cuda")
        pick += (torch.arange(H, device="cuda") * c["centres"]).view(1, H, 1)
        x = torch.randn(B, H, N, D, generator=g, device="cuda") * 0.5
        return (x + centre[pick]).to(dt)

    if c["op"].startswith("mixer"):
        C = H * D
        x = {"X": normal(B, N, C), "W_in": normal(c["n_proj"] * C, C, std=C ** -0.5),
             "Wo": normal(C, C, std=C ** -0.5), "seeds": normal(H, M, D)}
        if c["op"] == "mixer_train":
            x["dO"] = normal(B, N, C)
        return x
    x = {"seeds": normal(H, M, D)}
    if c["op"] != "flare":
        x["Kt"], x["Vt"] = keys(), normal(B, H, N, D)
    x["K"], x["V"] = keys(), normal(B, H, N, D)
    if c["op"] == "train":
        x["dY"] = normal(B, H, N, D)
    return x


def prepare(case, seed):
    # the forward's and the backward's workspaces: a program keeps one for each
    return {"op": case["op"], "scale": _scale(case), "x": _inputs(case, seed),
            "ws": flarepp.Workspace(), "ws_bwd": flarepp.Workspace()}


def run(state):
    x, s, ws = state["x"], state["scale"], state["ws"]
    op = state["op"]
    if op == "chain":
        return flarepp.route_fwd(x["seeds"], x["Kt"], x["Vt"], x["K"], x["V"], s, workspace=ws)
    if op == "flare":
        return flarepp.flare_fwd(x["seeds"], x["K"], x["V"], s, workspace=ws)
    if op == "train":
        a = (x["seeds"], x["Kt"], x["Vt"], x["K"], x["V"])
        Y, saved = flarepp.route_fwd_train(*a, s, workspace=ws)
        g = flarepp.route_bwd(*a, Y, x["dY"], saved, s, workspace=state["ws_bwd"])
        return dict(zip(("Y", "dseeds", "dKt", "dVt", "dK", "dV"), (Y, *g)))
    a = (x["X"], x["W_in"], x["Wo"], x["seeds"])
    if op == "mixer":
        return flarepp.mixer_fwd(*a, s, workspace=ws)
    O, saved = flarepp.mixer_fwd_train(*a, s, workspace=ws)
    g = flarepp.mixer_bwd(*a, saved, x["dO"], s, workspace=state["ws_bwd"])
    return dict(zip(("O", "dX", "dW_in", "dWo", "dseeds"), (O, *g)))


def work(case):
    """Each input read once, each output written once; the products of the three (FLARE: two)
    attention calls (4 flops per score and channel forward, 10 backward with the scores formed
    again) and of the projections."""
    B, H, N, M, D, op = (case[k] for k in ("B", "H", "N", "M", "D", "op"))
    e = 4 if case["dtype"] == "f32" else 2
    tok, seeds, C = B * H * N * D, H * M * D, H * D
    att = B * H * N * M * D
    if op == "chain":
        return {"bytes": e * (5 * tok + seeds), "flops": 12 * att}
    if op == "flare":
        return {"bytes": e * (3 * tok + seeds), "flops": 8 * att}
    if op == "train":
        return {"bytes": e * (10 * tok + 2 * seeds), "flops": 42 * att}
    w = (case["n_proj"] + 1) * C * C
    proj = 2 * B * N * w
    if op == "mixer":
        return {"bytes": e * (2 * tok + w + seeds), "flops": 12 * att + proj}
    return {"bytes": e * (4 * tok + 2 * w + 2 * seeds), "flops": 42 * att + 3 * proj}


# ------------------------------------------------------------------ the same in 64 bits

def _sdpa(a, b, c, s):
    """softmax(s a b^T) c and the row probabilities."""
    p = torch.softmax((a @ b.transpose(-1, -2)).mul_(s), dim=-1)
    return p @ c, p


def _sdpa_bwd(a, b, c, s, p, do):
    """Gradients of _sdpa's output for do: of a, b and c."""
    dc = p.transpose(-1, -2) @ do
    ds = do @ c.transpose(-1, -2)
    ds -= (do * (p @ c)).sum(-1, keepdim=True)
    ds *= p
    ds *= s
    return ds @ b, ds.transpose(-1, -2) @ a, dc


def _chain64(seeds, Kt, Vt, K, V, s, dY=None):
    """The chain of all (b, h) in float64, one (b, h) at a time: Y, and with dY the gradients."""
    B, H = K.shape[:2]
    Y = torch.empty(K.shape, dtype=torch.float64, device=K.device)
    g = None
    if dY is not None:
        g = [torch.zeros(t.shape, dtype=torch.float64, device=K.device)
             for t in (seeds, Kt, Vt, K, V)]
    for b in range(B):
        for h in range(H):
            q0, kt, vt, k, v = (t.double() for t in (seeds[h], Kt[b, h], Vt[b, h], K[b, h], V[b, h]))
            q, p1 = _sdpa(q0, kt, vt, s)
            if dY is None:
                del p1
            z, p2 = _sdpa(q, k, v, s)
            if dY is None:
                del p2
            Y[b, h], p3 = _sdpa(k, q, z, s)
            if dY is None:
                continue
            dk, dq, dz = _sdpa_bwd(k, q, z, s, p3, dY[b, h].double())
            del p3
            dq2, dk2, dv = _sdpa_bwd(q, k, v, s, p2, dz)
            del p2
            d0, dkt, dvt = _sdpa_bwd(q0, kt, vt, s, p1, dq + dq2)
            del p1
            g[0][h] += d0
            for t, x in zip(g[1:], (dkt, dvt, dk + dk2, dv)):
                t[b, h] = x
    return Y, g


def exact(case, seed):
    x, s = _inputs(case, seed), _scale(case)
    op = case["op"]
    if op == "flare":
        q, k, v = x["seeds"].double(), x["K"], x["V"]
        Y = torch.empty(k.shape, dtype=torch.float64, device=k.device)
        for b in range(case["B"]):
            kb, vb = k[b].double(), v[b].double()
            z, _ = _sdpa(q, kb, vb, s)
            Y[b], _ = _sdpa(kb, q, z, s)
        return Y
    if op in ("chain", "train"):
        Y, g = _chain64(x["seeds"], x["Kt"], x["Vt"], x["K"], x["V"], s, x.get("dY"))
        return Y if g is None else dict(zip(("Y", "dseeds", "dKt", "dVt", "dK", "dV"), (Y, *g)))
    B, H, N, D, P = case["B"], case["H"], case["N"], case["D"], case["n_proj"]
    X, W, Wo = x["X"].double(), x["W_in"].double(), x["Wo"].double()
    C = H * D

    def split(t):  # [B, N, C] -> [B, H, N, D]
        return t.view(B, N, H, D).transpose(1, 2).contiguous()

    def merge(t):
        return t.transpose(1, 2).reshape(B, N, C)

    heads = [split(X @ W[p * C:(p + 1) * C].T) for p in range(P)]
    K, V = heads[0], heads[1]
    Kt, Vt = (heads[2], heads[3]) if P == 4 else (K, V)
    dO = x["dO"].double() if op == "mixer_train" else None
    Y, g = _chain64(x["seeds"], Kt, Vt, K, V, s, None if dO is None else split(dO @ Wo))
    O = merge(Y) @ Wo.T
    if dO is None:
        return O
    d0, dKt, dVt, dK, dV = g
    d = [dK, dV, dKt, dVt] if P == 4 else [dK + dKt, dV + dVt]
    flat = [merge(t).view(B * N, C) for t in d]
    dX = sum(f @ W[p * C:(p + 1) * C] for p, f in enumerate(flat)).view(B, N, C)
    dW = torch.cat([f.T @ X.view(B * N, C) for f in flat])
    dWo = dO.view(B * N, C).T @ merge(Y).view(B * N, C)
    return {"O": O, "dX": dX, "dW_in": dW, "dWo": dWo, "dseeds": d0}
