"""The barrier protocol of the token passes (tc_tok.cu), checked as a model on the CPU.

One CTA's roles follow the kernel's waits, arrivals and commits: the TMA producer, the MMA issuer and four
softmax warpgroups (two per stream; a warpgroup's 128 threads arrive together). TMA copies complete in any
order, products and commits in the order they are issued, everything else in random order, also with one
role slowed to one step in fifty. Waits are taken by phase parity, as the hardware takes them. The model
fails on deadlock, when a barrier is two phases ahead of a waiter or behind the phase it names, and when a
product, a copy or a softmax step finds a ring stage, a token tile, a score tile, a dS tile or an
accumulator holding other data than it is for, or still in use. Planted mistakes are caught."""
import random

import pytest


class Bar:
    def __init__(self, count):
        self.count, self.left, self.phase = count, count, 0

    def arrive(self):
        self.left -= 1
        assert self.left >= 0
        if self.left == 0:
            self.phase, self.left = self.phase + 1, self.count


class Model:
    """segments: token tiles of each (b, h) segment in turn; n_items: route items of 64."""

    def __init__(self, rng, segments, n_items, stages, call1, slow=None, mistake=None):
        self.rng, self.n_items, self.S, self.call1 = rng, n_items, stages, call1
        self.slow, self.mistake = slow, mistake
        self.tiles = [(seg, k == n - 1) for seg, n in enumerate(segments) for k in range(n)]
        self.nb = (n_items + 1) // 2
        B = Bar
        self.full = [B(1) for _ in range(stages)]
        self.empty = [B(1) for _ in range(stages)]
        self.afull, self.aready, self.afree = ([B(c) for _ in range(2)] for c in (1, 4, 1))
        self.sready, self.pready = ([B(c) for _ in range(2)] for c in (1, 2))
        self.accdone, self.accfree = ([B(c) for _ in range(2)] for c in (1, 4))
        self.statfull, self.segfree, self.dqdone = [B(1), B(1)], [B(4), B(4)], B(1)
        # what the buffers hold, and how many uses of it are still to come
        self.ring, self.ring_uses = [None] * stages, [0] * stages
        self.tile, self.tile_uses, self.scaled = [None] * 2, [0] * 2, [0] * 2
        self.stat = [None] * 2
        self.sc, self.sc_unread = [None] * 2, [0] * 2     # S and T of a stream; readers to come
        self.p, self.ds, self.ds_uses = [0] * 2, {}, {}   # P halves written; dS [buffer, stream]
        self.acc, self.acc_unread = [None] * 2, [0] * 2   # dK, dV by tile parity
        self.dq, self.dq_unread = None, 0
        self.copies, self.mma = [], []

    # ------------------------------------------------------------ waits by parity
    def ready(self, bar, n):
        assert bar.phase - n in (0, 1), "a barrier two phases away from a waiter"
        return bar.phase == n + 1

    def wait(self, bar, n):
        while not self.ready(bar, n):
            yield False
        yield True

    # ------------------------------------------------------------ roles
    def producer(self):
        it, seg = 0, -1
        for tc, (sg, _) in enumerate(self.tiles):
            if sg != seg:
                seg, b = sg, sg & 1
                if sg >= 2:
                    yield from self.wait(self.segfree[b], (sg >> 1) - 1)
                self.stat[b] = sg
                self.statfull[b].arrive()
            b = tc & 1
            if tc >= 2 and self.mistake != "no afree":
                yield from self.wait(self.afree[b], (tc >> 1) - 1)
            assert self.tile_uses[b] == 0, "a token tile is overwritten in use"
            # uses: K by every S and dQ, the tile as a whole
            self.tile[b], self.scaled[b] = None, 0
            self.tile_uses[b] = 2 * self.n_items + self.nb
            self.copies.append(("tile", b, tc))
            for i in range(self.n_items):
                st = it % self.S
                if it >= self.S:
                    yield from self.wait(self.empty[st], it // self.S - 1)
                assert self.ring_uses[st] == 0, "a ring stage is overwritten in use"
                self.ring[st], self.ring_uses[st] = None, 4  # S, T, dV, dK
                self.copies.append(("item", st, (tc, i)))
                it += 1
                yield True

    def issuer(self):
        it, n_s, bg, n_fresh, fresh = 0, [0, 0], 0, 0, True
        o = None

        def wait_owed(s):
            yield from self.wait(self.pready[s], n_s[s] - 1)
            if s == 0 and o["first"] and o["tc"] >= 2 and self.mistake != "no accfree":
                yield from self.wait(self.accfree[o["tc"] & 1], (o["tc"] >> 1) - 1)

        def turn(s, item, st):
            owed = o is not None and (s == 0 or o["two"])
            if item is not None:
                self.mma.append(("S", s, item, st))
            if owed:
                self.mma.append(("dV", s, o, bg))
            if item is not None:
                self.mma.append(("T", s, item, st))
                self.mma.append(("commit", self.sready[s]))
            if owed:
                self.mma.append(("dK", s, o, bg))
                self.mma.append(("commit", self.empty[o["st"][s]]))

        def finish_block():
            self.mma.append(("dQ", o, bg))
            if o["last"]:
                self.mma.append(("commit", self.afree[o["tc"] & 1]))
                self.mma.append(("commit", self.accdone[o["tc"] & 1]))
                if o["seg_end"]:
                    self.mma.append(("commit", self.dqdone))

        def wait_dq():
            nonlocal n_fresh
            if o["fresh"] and o["first"]:
                n_fresh += 1
                if n_fresh > 1 and self.mistake != "no segfree":
                    yield from self.wait(self.segfree[(n_fresh - 2) & 1], (n_fresh - 2) >> 1)

        for tc, (sg, seg_end) in enumerate(self.tiles):
            yield from self.wait((self.afull if self.call1 else self.aready)[tc & 1], tc >> 1)
            for b in range(self.nb):
                has1 = 2 * b + 1 < self.n_items
                st = (it % self.S, (it + 1) % self.S)
                yield from self.wait(self.full[st[0]], it // self.S)
                if o:
                    yield from wait_owed(0)
                turn(0, (tc, 2 * b), st[0])
                n_s[0] += 1
                if has1:
                    yield from self.wait(self.full[st[1]], (it + 1) // self.S)
                if o and o["two"]:
                    yield from wait_owed(1)
                turn(1, (tc, 2 * b + 1) if has1 else None, st[1])
                n_s[1] += has1
                it += 2 if has1 else 1
                if o:
                    yield from wait_dq()
                    finish_block()
                o = {"two": has1, "first": b == 0, "last": b + 1 == self.nb, "seg_end": seg_end, "fresh": fresh,
                     "tc": tc, "st": st, "b": b, "seg": sg}
                bg += 1
                yield True
            fresh = seg_end
        yield from wait_owed(0)
        turn(0, None, 0)
        if o["two"]:
            yield from wait_owed(1)
            turn(1, None, 0)
        yield from wait_dq()
        finish_block()

    def softmax(self, w):
        s = w >> 1
        n_is, bg, n_epi, seg, owed = 0, 0, 0, -1, None
        prep_at = self.nb - 2 if self.nb > 1 else 0

        def prep(tc):
            if self.call1:
                return
            yield from self.wait(self.afull[tc & 1], tc >> 1)
            assert self.tile[tc & 1] == tc, "V is scaled in another tile"
            self.scaled[tc & 1] += 1
            self.aready[tc & 1].arrive()

        def read_acc():
            nonlocal n_epi
            par = n_epi & 1
            yield from self.wait(self.accdone[par], n_epi >> 1)
            assert self.acc[par] == owed and self.acc_unread[par] > 0, "accumulators of another tile"
            self.acc_unread[par] -= 1
            self.accfree[par].arrive()
            n_epi += 1

        yield from prep(0)
        for tc, (sg, seg_end) in enumerate(self.tiles):
            if sg != seg:
                seg = sg
                yield from self.wait(self.statfull[sg & 1], sg >> 1)
            for b in range(self.nb):
                item = 2 * b + s
                if item < self.n_items:
                    yield from self.wait(self.sready[s], n_is)
                    n_is += 1
                    assert self.sc[s] == (tc, item), "another item's scores"
                    assert self.stat[sg & 1] == sg, "another segment's statistics"
                    self.sc_unread[s] -= 1
                    buf = ((bg if self.mistake != "one dS buffer" else 0) & 1, s)
                    if self.ds.get(buf) != (tc, item):
                        assert self.ds_uses.get(buf, 0) == 0, "dS is overwritten in use"
                        self.ds[buf], self.ds_uses[buf] = (tc, item), 2  # dK, dQ
                    yield True
                    self.p[s] += 1
                    self.pready[s].arrive()
                    if owed is not None:
                        yield from read_acc()
                        owed = None
                if b == prep_at and tc + 1 < len(self.tiles):
                    yield from prep(tc + 1)
                bg += 1
            if owed is not None:
                yield from read_acc()
            owed = tc
            if seg_end:
                yield from self.wait(self.dqdone, sg)
                assert self.dq == sg and self.dq_unread > 0, "dQ of another segment"
                self.dq_unread -= 1
                self.segfree[sg & 1].arrive()
        yield from read_acc()

    # ------------------------------------------------------------ the tensor pipe and the copies
    def use_item(self, st, item):
        assert self.ring[st] == item, "a product reads another item"
        self.ring_uses[st] -= 1

    def use_tile(self, tc):
        assert self.tile[tc & 1] == tc, "a product reads another token tile"
        self.tile_uses[tc & 1] -= 1

    def execute(self, op):
        kind = op[0]
        if kind == "commit":
            op[1].arrive()
        elif kind in ("S", "T"):
            _, s, item, st = op
            self.use_tile(item[0])
            self.use_item(st, item)
            if kind == "S":
                assert self.sc_unread[s] == 0, "scores are overwritten unread"
                self.sc[s] = None
            else:
                assert self.call1 or self.scaled[item[0] & 1] == 4, "T before V is scaled"
                assert self.p[s] == 0, "T overwrites P"
                self.sc[s], self.sc_unread[s] = item, 2
        elif kind in ("dV", "dK"):
            _, s, o, bg = op
            item, par = (o["tc"], 2 * o["b"] + s), o["tc"] & 1
            self.use_item(o["st"][s], item)
            if kind == "dV":
                assert self.p[s] == 2, "dV without P"
                self.p[s] = 0
                if o["first"] and s == 0:
                    assert self.acc_unread[par] == 0, "accumulators are started unread"
                    self.acc[par] = o["tc"]
                assert self.acc[par] == o["tc"]
            else:
                self.use_ds(bg, s, item)
        else:
            _, o, bg = op
            for s in range(2 if o["two"] else 1):
                self.use_ds(bg, s, (o["tc"], 2 * o["b"] + s))
            self.use_tile(o["tc"])
            if o["fresh"] and o["first"]:
                assert self.dq_unread == 0, "dQ is started unread"
                self.dq = o["seg"]
            assert self.dq == o["seg"]
            if o["last"]:
                self.acc_unread[o["tc"] & 1] = 4
                if o["seg_end"]:
                    self.dq_unread = 4

    def use_ds(self, bg, s, item):
        buf = ((bg - 1 if self.mistake != "one dS buffer" else 0) & 1, s)
        assert self.ds.get(buf) == item, "a product reads another item's dS"
        self.ds_uses[buf] -= 1

    def run(self):
        roles = {"producer": self.producer(), "issuer": self.issuer()}
        roles.update({f"softmax{w}": self.softmax(w) for w in range(4)})
        idle = 0
        while roles or self.copies or self.mma:
            choices = [("role", r) for r in roles if r != self.slow or self.rng.random() < 0.02]
            choices += [("copy", k) for k in range(len(self.copies))]
            if self.mma:
                choices.append(("mma", 0))
            if not choices:
                continue
            kind, k = self.rng.choice(choices)
            if kind == "copy":
                what, b, content = self.copies.pop(k)
                if what == "tile":
                    self.tile[b] = content
                    self.afull[b].arrive()
                else:
                    self.ring[b] = content
                    self.full[b].arrive()
                idle = 0
            elif kind == "mma":
                self.execute(self.mma.pop(0))
                idle = 0
            else:
                try:
                    idle = 0 if next(roles[k]) else idle + 1
                except StopIteration:
                    del roles[k]
                    idle = 0
            assert idle < 20000 or self.copies or self.mma, "deadlock"


SEGMENTS = [[1], [2], [5], [1, 1, 1, 1], [2, 1, 3], [1, 4, 1, 1, 2]]


@pytest.mark.parametrize("slow", [None, "producer", "issuer", "softmax0", "softmax3"])
@pytest.mark.parametrize("call1,stages", [(False, 5), (False, 6), (True, 6)])
@pytest.mark.parametrize("n_items", [1, 2, 3, 5, 8])
def test_token_pass_protocol(n_items, call1, stages, slow):
    for seed, segments in enumerate(SEGMENTS):
        Model(random.Random(seed), segments, n_items, stages, call1, slow).run()


@pytest.mark.parametrize("mistake,call1,n_items", [
    ("no afree", False, 2), ("no accfree", True, 2), ("no segfree", True, 1), ("one dS buffer", False, 2),
    ("one dS buffer", True, 2)])
def test_planted_mistakes_are_caught(mistake, call1, n_items):
    """(In calls 3 and 2 the wait for the scaled V, to which every softmax warp arrives late in the tile before,
    implies the waits that are left out in call 1 alone; with two streams at work in a block, so do their P.)"""
    caught = 0
    for seed in range(40):
        for slow in (None, "softmax0", "softmax3", "issuer"):
            try:
                Model(random.Random(seed), [1, 1, 3, 1, 2], n_items, 6, call1, slow, mistake).run()
            except AssertionError:
                caught += 1
    assert caught > 0
