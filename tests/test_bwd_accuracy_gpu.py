"""How exact the gradients of call 1 are on the token passes that form dQ (tc_tok.cu).

dQ takes dP2 = V dZ^T, a difference of large terms when the values share an offset: call 2's
dS2 = P2 (dP2 - <dZ, Z>) sees V only through V - Z. V itself is exact in bf16, but the pass multiplies
it with the row factor u = 2^(L3 - R), and u V rounded to one bf16 would bring back an error of 2^-9 of
the offset. So u V is taken as a pair of bf16 operands. Here V sits at `offset` and dY at `lean` (so that
dZ, and with it call 2's share of dQ, is large).

The reference is the backward alone in float64 (App. A.5), of the values that the training forward gave:
its saved Q and Z (in the operands' form: Q as a bf16 pair in the scores, Z in bf16), its
log-normalisers and its Y. (The forward's own rounding of P2 moves Z, and with offset values the
gradients of the exact chain by up to 1.4e-2: that is no part of the backward.)

Bounds, on the root mean square of the error over that of the gradient: dQ and each gradient are rounded
to bf16 once (2^-9 times 0.85 each, the rms of a rounding over a uniform mantissa), as are P1, dS and
w dZ ahead of sums that average them; dVt sees two of these in full, dKt and dseeds also the rounding of
dS1, which a difference with c1 magnifies (dseeds sums them over the tokens): 2^-8 for dVt, 2^-7 for dKt,
1e-2 for dseeds. With u V rounded once all three miss them (1.2e-2 at least in an emulation)."""
import math

import pytest
import torch

from paper_2608_11519_gb300 import flarepp

pytestmark = pytest.mark.gpu

BOUND = {"dseeds": 1e-2, "dKt": 2.0 ** -7, "dVt": 2.0 ** -8}

CASES = [  # N, M, D, centres, scale, offset, lean
    (4000, 16, 16, 0, 0.1, 8.0, 2.0),
    (4000, 32, 32, 64, 0.05, 4.0, 1.0),
]


def make_inputs(N, M, D, centres, offset, lean, H=2):
    g = torch.Generator().manual_seed(17)

    def normal(*shape):
        return torch.randn(*shape, generator=g)

    def keys():
        if not centres:
            return normal(1, H, N, D)
        centre = 1.5 * normal(H, centres, D)
        pick = torch.randint(0, centres, (H, N), generator=g)
        return (0.5 * normal(H, N, D) + torch.stack([centre[h, pick[h]] for h in range(H)]))[None]

    x = {"seeds": normal(H, M, D), "Kt": keys(), "Vt": normal(1, H, N, D), "K": keys(),
         "V": offset + normal(1, H, N, D), "dY": lean + normal(1, H, N, D)}
    return {k: v.to(torch.bfloat16) for k, v in x.items()}


def _bf16(t):
    return t.to(torch.bfloat16).double()


def _saved(saved, H, N, M, D):
    """Q, Z [H, M, D], L1, L2 [H, M], L3 [H, N] of the training forward's state (blocks of 256 bytes)."""
    out, off = [], 0
    for shape in ((H, M, D), (H, M, D), (H, M), (H, M), (H, N)):
        n = 4 * math.prod(shape)
        out.append(saved[off:off + n].view(torch.float32).view(shape))
        off += (n + 255) // 256 * 256
    return out


def backward64(x, Y, saved, scale):
    seeds, Kt, Vt, K, V, dY = (x[k].double().reshape(x["seeds"].shape[0], -1, x["K"].shape[-1])
                               for k in ("seeds", "Kt", "Vt", "K", "V", "dY"))
    Q32, Z32, L1, L2, L3 = _saved(saved, seeds.shape[0], K.shape[1], seeds.shape[1], K.shape[2])
    Q = _bf16(Q32) + _bf16(Q32 - Q32.to(torch.bfloat16).float())
    Z = _bf16(Z32)
    L1, L2, L3 = L1.double(), L2.double(), L3.double()
    c = scale / math.log(2.0)
    T = lambda t: t.transpose(-1, -2)
    S = c * K @ T(Q)  # [H, N, M]
    P3 = torch.exp2(S - L3[..., None])
    dS3 = P3 * (dY @ T(Z) - (dY * Y.double()[0]).sum(-1, keepdim=True))
    dZ = T(P3) @ dY
    P2 = torch.exp2(S - L2[:, None, :])
    dS2 = P2 * (V @ T(dZ) - (dZ * Z32.double()).sum(-1)[:, None, :])
    dQ = scale * (T(dS3 + dS2) @ K)
    P1 = torch.exp2(c * Kt @ T(seeds) - L1[:, None, :])
    dS1 = P1 * (Vt @ T(dQ) - (dQ * Q32.double()).sum(-1)[:, None, :])
    return {"dseeds": scale * (T(dS1) @ Kt), "dKt": (scale * dS1 @ seeds)[None], "dVt": (P1 @ dQ)[None]}


@pytest.mark.parametrize("N,M,D,centres,scale,offset,lean", CASES)
def test_gradients_of_call_1_with_offset_values(N, M, D, centres, scale, offset, lean):
    x = {k: v.cuda() for k, v in make_inputs(N, M, D, centres, offset, lean).items()}
    args = tuple(x[k] for k in ("seeds", "Kt", "Vt", "K", "V"))
    Y, saved = flarepp.route_fwd_train(*args, scale)
    got = dict(zip(("dseeds", "dKt", "dVt", "dK", "dV"),
                   flarepp.route_bwd(*args, Y, x["dY"], saved, scale)))
    want = backward64(x, Y, saved, scale)
    for name, bound in BOUND.items():
        err = float((got[name].double() - want[name]).norm() / want[name].norm())
        assert err <= bound, f"{name}: {err} > {bound}"


def test_float32_sums_over_many_tokens():
    """The float32 route passes sum at most 256 tokens in a register before they add to the chunk's partial.
    With one route P3 = 1, dZ is the sum of dY over the tokens and dV_n = P2_n dZ: the direction of dV_n is
    that of dZ, whatever the error of P2. 1,216 heads leave one chunk of 1,500 tokens to each. dY = 1 + noise
    added up in one float32 chain has an error of sqrt(1500 / 3) 2^-24 0.41 = 5.4e-7 rms (every sum so far
    rounded once), in parts of 256 2.2e-7 and 0.9e-7 for adding the parts; the product with P2 adds 0.2e-7.
    The bound is the geometric mean of 5.4e-7 and 2.4e-7."""
    B, H, N, M, D = 152, 8, 1500, 1, 32
    g = torch.Generator(device="cuda").manual_seed(3)

    def normal(*shape):
        return torch.randn(*shape, generator=g, device="cuda")

    scale = D ** -0.5
    args = (normal(H, M, D), normal(B, H, N, D), normal(B, H, N, D), normal(B, H, N, D), normal(B, H, N, D))
    dY = 1.0 + 0.25 * normal(B, H, N, D)
    Y, saved = flarepp.route_fwd_train(*args, scale)
    dV = flarepp.route_bwd(*args, Y, dY, saved, scale)[4].double()
    want = dY.double().sum(2, keepdim=True)
    want = want / want.norm(dim=-1, keepdim=True)
    err = float((dV / dV.norm(dim=-1, keepdim=True) - want).pow(2).sum(-1).mean().sqrt())
    assert err <= 3.6e-7, err
