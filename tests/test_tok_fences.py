"""Tensor memory changes hands in the token passes (tc_tok.cu) by mbarriers, and an mbarrier alone does not
order tcgen05 instructions: whoever takes columns over after a wait needs a tcgen05
fence::after_thread_sync before its next tcgen05 instruction, as whoever gives them away needs a
fence::before_thread_sync before it arrives. A missing one may never show in a result, so the order is
checked in the source: in the issuer's role every wait for threads that read or write TMEM (the softmax
warps' P and dS, the accumulators read out, dQ given back) is followed by the fence before the next
product, and in the softmax role by the fence before the next TMEM load."""
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                   "paper_2608_11519_gb300", "csrc", "tc_tok.cu")


def _roles():
    text = open(SRC).read()
    marks = [text.index(m) for m in ("- MMA issuer", "- softmax warpgroups", "- host side")]
    return [re.sub(r"//[^\n]*", "", text[a:b]) for a, b in zip(marks, marks[1:])]


def _block(text, at):
    """The {...} block that opens at or after `at`, and where it ends."""
    first = text.index("{", at)
    depth = 0
    for i in range(first, len(text)):
        depth += {"{": 1, "}": -1}.get(text[i], 0)
        if depth == 0:
            return text[first:i + 1], i + 1
    raise AssertionError("unbalanced braces")


def _inline(text, names):
    """The text with the bodies of the named lambdas in place of their calls."""
    bodies = {}
    for n in names:
        at = text.index(f"auto {n} = [&]")
        body, end = _block(text, text.index(")", at))
        bodies[n] = body
        text = text[:at] + text[end:]
    for n, body in bodies.items():
        text = re.sub(rf"\b{n}\(", lambda m: f" {body} {m.group(0)}", text)
    return text


def _check(text, waits, uses):
    token = re.compile(rf"wait\((?P<w>{waits})\b|(?P<f>tc_fence_after\()|\b(?P<u>{uses})\(")
    pending, seen = None, 0
    for m in token.finditer(text):
        if m.group("w"):
            pending = m.group("w")
            seen += 1
        elif m.group("f"):
            pending = None
        else:
            assert pending is None, f"{m.group('u')} after a wait on {pending} without the fence"
    return seen


def test_issuer_fences_after_every_handover():
    issuer, _ = _roles()
    turn_at = issuer.index("auto turn = [&]")
    _, end = _block(issuer, issuer.index(")", turn_at))
    issuer = issuer[:turn_at] + issuer[end:]  # (the products themselves)
    at = issuer.index("auto finish_block = [&]")
    _, end = _block(issuer, issuer.index(")", at))
    issuer = issuer[:at] + issuer[end:]
    flat = _inline(issuer, ("wait_owed", "wait_dq"))
    assert _check(flat, "pready0|accfree0|segfree0", "turn|finish_block") >= 10


def test_softmax_fences_after_every_handover():
    _, soft = _roles()
    assert _check(soft, "sready0|accdone0|dqdone", "tmem_ld16|tmem_ld8|tmem_st8") >= 3
