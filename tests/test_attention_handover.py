"""The hand-overs of the prefill attention kernel (csrc/attention.cu), run through a model on the CPU: one generator per role (loads and items, scores,
products, eight softmax warps, where rows are fetched by index a second loading warp), barriers that show one bit of their phase, loads that land in any order, products and commits that complete in the
order in which their thread issued them, at any time.  Every buffer carries what was put into it and every reader checks it; a state in
which nothing can move is an error."""
import itertools
import random

import pytest

K_SLOTS, V_SLOTS, RECORDS = 3, 2, 4


class Bar:
    def __init__(self, count):
        self.count, self.left, self.phase = count, count, 0

    def arrive(self):
        self.left -= 1
        if self.left == 0:
            self.left, self.phase = self.count, self.phase + 1

    def passed(self, parity):
        return (self.phase & 1) != parity


class Model:
    """items: (pair, top), top the number of the highest query tile, key blocks 0 .. top; a pair has tile top - 1 as well."""

    def __init__(self, items, rng, wait_free=True, helper=False):
        self.helper, self.parts = helper, {}
        self.items, self.rng, self.wait_free, self.ragged = items, rng, wait_free, [rng.random() < 0.7 for _ in items]
        two = lambda c: [Bar(c), Bar(c)]
        self.q_full, self.q_free, self.s_full, self.s_free, self.p_full, self.o_full = two(1), two(1), two(1), two(4), two(4), two(1)
        self.k_full, self.k_free = [Bar(1) for _ in range(K_SLOTS)], [Bar(1) for _ in range(K_SLOTS)]
        self.v_full, self.v_free = [Bar(1) for _ in range(V_SLOTS)], [Bar(1) for _ in range(V_SLOTS)]
        self.i_full, self.i_free = [Bar(1) for _ in range(RECORDS)], [Bar(10 + helper) for _ in range(RECORDS)]
        self.rec, self.q, self.k, self.v = [None] * RECORDS, [None] * 2, [None] * K_SLOTS, [None] * V_SLOTS
        self.cleared = [0] * V_SLOTS
        self.s, self.s_readers, self.p, self.o = None, 0, [[None] * 4, [None] * 4], [None] * 2
        self.landing, self.pipe = [], {"score": [], "product": []}
        self.haste = {id(buf): rng.choice([1, 1, 30]) for buf in (self.q, self.k, self.v)}
        self.done = []

    # -- asynchronous work --
    def load(self, buf, slot, what, full):
        buf[slot] = "in flight"
        self.landing.append((buf, slot, what, full))

    def land(self):
        at = self.rng.choices(range(len(self.landing)), [self.haste[id(e[0])] for e in self.landing])[0]
        buf, slot, what, full = self.landing.pop(at)
        if self.helper:                                 # a tile is there when both warps' halves are
            parts = self.parts.setdefault((id(buf), slot), [])
            parts.append(what)
            assert parts.count(what) == len(parts)
            if len(parts) < 2:
                return
            parts.clear()
        buf[slot] = what
        if buf is self.v:
            self.cleared[slot] = 0
        full.arrive()

    # -- roles --
    def loader(self, helps=False):
        kf = vf = turn = 0
        qn = [0, 0]

        def q(x, what):
            yield self.q_free[x], (qn[x] & 1) ^ 1
            qn[x] += 1
            self.load(self.q, x, what, self.q_full[x])

        for n, (pair, top) in enumerate(self.items + [(False, -1)]):
            slot = n % RECORDS
            if helps:
                _, top, first, last = yield from self.next_item(n)
                pair = first < last
            else:
                yield self.i_free[slot], ((n // RECORDS) & 1) ^ 1
                pair = pair and top > 0
                first, last = (0, 1) if pair else (turn, turn)
                turn = 0 if pair else turn ^ 1
                self.rec[slot] = (n, top, first, last)
                self.i_full[slot].arrive()
            if top < 0:
                return
            if pair:
                yield from q(0, (n, top - 1))
            for t in range(top + 2):
                if t <= top:
                    yield self.k_free[kf % K_SLOTS], ((kf // K_SLOTS) & 1) ^ 1
                    self.load(self.k, kf % K_SLOTS, (n, t), self.k_full[kf % K_SLOTS])
                    kf += 1
                if t == 0:
                    yield from q(last, (n, top))
                else:
                    yield self.v_free[vf % V_SLOTS], ((vf // V_SLOTS) & 1) ^ 1
                    self.load(self.v, vf % V_SLOTS, (n, t - 1), self.v_full[vf % V_SLOTS])
                    vf += 1

    def next_item(self, n):
        slot = n % RECORDS
        yield self.i_full[slot], (n // RECORDS) & 1
        rec = self.rec[slot]
        assert rec[0] == n
        self.i_free[slot].arrive()
        return rec

    def score(self):
        used, holder, made, qn = 0, None, [0, 0], [0, 0]
        pipe = self.pipe["score"]
        for n in itertools.count():
            _, top, first, last = yield from self.next_item(n)
            if top < 0:
                return
            for j in range(top + 1):
                ks = used % K_SLOTS
                yield self.k_full[ks], (used // K_SLOTS) & 1
                for x in range(first if j < top else last, last + 1):
                    if j == 0:
                        yield self.q_full[x], qn[x] & 1
                    if holder is not None:
                        yield self.s_free[holder], (made[holder] & 1) ^ 1
                    pipe.append(("S", x, ks, (n, j), (n, top - (last - x))))
                    pipe.append(("commit", self.s_full[x]))
                    made[x] += 1
                    holder = x
                    if j == top - (last - x):
                        pipe.append(("commit", self.q_free[x]))
                        qn[x] += 1
                pipe.append(("commit", self.k_free[ks]))
                used += 1

    def product(self):
        used, pn = 0, [0, 0]
        pipe = self.pipe["product"]
        for n in itertools.count():
            _, top, first, last = yield from self.next_item(n)
            if top < 0:
                return
            for j in range(top + 1):
                vs = used % V_SLOTS
                yield self.v_full[vs], (used // V_SLOTS) & 1
                for x in range(first if j < top else last, last + 1):
                    yield self.p_full[x], pn[x] & 1
                    pn[x] += 1
                    pipe.append(("O", x, vs, (n, j), j == top and self.ragged[n]))
                    pipe.append(("commit", self.o_full[x]))
                pipe.append(("commit", self.v_free[vs]))
                used += 1

    def complete(self, role):
        op = self.pipe[role].pop(0)
        if op[0] == "commit":
            op[1].arrive()
        elif op[0] == "S":
            _, x, ks, what, tile = op
            assert self.k[ks] == what and self.q[x] == tile and self.s_readers == 0
            self.s, self.s_readers = (x, what), 4
        else:
            _, x, vs, what, ragged = op
            assert self.v[vs] == what and self.p[x] == [what] * 4
            assert not ragged or self.cleared[vs] == 4, "a product has read rows that were not cleared"
            assert self.o[x] == (what[0], what[1] - 1) or what[1] == 0
            self.o[x] = what

    def softmax(self, x, w):
        blocks = v_blocks = 0
        for n in itertools.count():
            _, top, first, last = yield from self.next_item(n)
            if top < 0:
                return
            v_first, v_blocks = v_blocks, v_blocks + top + 1
            if not first <= x <= last:
                continue
            qt = top - (last - x)
            for j in range(qt + 1):
                yield self.s_full[x], blocks & 1
                assert self.s == (x, (n, j))
                self.s_readers -= 1
                self.s_free[x].arrive()
                if j > 0:
                    yield self.o_full[x], (blocks - 1) & 1
                    assert self.o[x] == (n, j - 1)
                self.p[x][w] = (n, j)
                if j == qt and x == last and self.ragged[n]:
                    vb = v_first + j
                    vs, use = vb % V_SLOTS, vb // V_SLOTS
                    if j == 0 and use and self.wait_free:
                        yield self.v_free[vs], (use - 1) & 1
                    yield self.v_full[vs], use & 1
                    assert self.v[vs] == (n, j), "cleared a tile that had not arrived"
                    self.cleared[vs] += 1
                self.p_full[x].arrive()
                blocks += 1
            yield self.o_full[x], (blocks - 1) & 1
            assert self.o[x] == (n, qt)
            if w == 0:
                self.done.append((n, qt))

    def run(self):
        roles = [self.loader()] + [self.loader(True)] * self.helper + [self.score(), self.product()] + [self.softmax(x, w) for x in range(2) for w in range(4)]
        waits = {g: None for g in roles}
        # speeds drawn anew for every run: some roles and kinds of work are much slower than others
        speed = {k: self.rng.choice([1, 1, 4, 30]) for k in [*roles, "land", "score", "product"]}
        while True:
            can = [g for g, w in waits.items() if w is None or w[0].passed(w[1])]
            can += ["land"] * bool(self.landing) + [r for r in ("score", "product") if self.pipe[r]]
            if not can:
                break
            g = self.rng.choices(can, [speed[c] for c in can])[0]
            if g == "land":
                self.land()
            elif isinstance(g, str):
                self.complete(g)
            else:
                try:
                    waits[g] = next(g)
                except StopIteration:
                    del waits[g]
        assert not waits, "stuck"
        tiles = {(n, t) for n, (pair, top) in enumerate(self.items) for t in ([top - 1, top] if pair and top else [top])}
        assert len(self.done) == len(tiles) and set(self.done) == tiles


def _mixes():
    rng = random.Random(1)
    forms = [(False, 0), (False, 1), (False, 2), (True, 1), (True, 2), (True, 3)]
    for length in (1, 2, 3):
        yield from (list(m) for m in itertools.product(forms, repeat=length))
    for _ in range(300):
        yield [(rng.random() < 0.5, min(int(rng.expovariate(0.6)), 6)) for _ in range(rng.randint(4, 12))]


@pytest.mark.parametrize("helper", [False, True], ids=["tiles", "rows by index"])
def test_no_mix_of_items_gets_stuck_or_reads_a_buffer_out_of_turn(helper):
    for n, items in enumerate(_mixes()):
        for s in range(3):
            Model(items, random.Random(1000 * n + s), helper=helper).run()


def test_the_model_sees_a_softmax_warp_that_takes_an_older_v_tile_for_its_own():
    with pytest.raises(AssertionError):
        for s in range(1000):
            Model([(False, 0), (False, 2)] * 4, random.Random(s), wait_free=False).run()
