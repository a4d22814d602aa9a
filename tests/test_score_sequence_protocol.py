"""Host models of the score passes' synchronisation over sequences of units
(score_lse_tc_kernel and score_colsum_tc_kernel, csrc/score_tc.cu).

test_score_protocol.py models one unit a pair; the passes are persistent.  With
the same engine (coroutines in the kernels' order, an in-order MMA pipe, unordered
copies, a random scheduler):

* pass 1 over a list of units (odd, even and no tiles): query rows double
  buffered across units, the warpgroups' use counts of their tensor-memory slots
  carried from unit to unit, and the exchange of statistics (warpgroup 1 arrives at
  half-full and syncs at half-empty, warpgroup 0 the other way round);
* pass 2 over the segments of several pairs that share units: slots by (layer,
  chunk), the double-buffered exchange of column sums, the sums a split unit
  leaves in memory, the counts that pass 1 clears, and the pair that comes last.

Planted mistakes (a missing wait, a single buffer, a count before its order) must
be caught.  No arithmetic is modelled."""
import pytest

from test_score_protocol import Engine, ProtocolError


def _caught(run):
    n = 0
    for seed in range(300):
        try:
            run(seed)
        except ProtocolError:
            n += 1
    return n


class Named:
    """A named barrier of two parties: sync = arrive and wait, or arrive alone."""

    def __init__(self, E, name):
        self.E, self.name = E, name
        E.bar(name, 2)
        self.round = {}

    def arrive(self, who):
        n = self.round.get(who, 0)
        self.round[who] = n + 1
        others = [r for w, r in self.round.items() if w != who]
        self.E.need(n <= (others[0] if others else 0), "%s arrives twice at %s" % (who, self.name))
        self.E.bars[self.name].arrive()
        return self.name, n


def run_pass1(units, seed, mistake=None):
    """One pair's units (tiles of each)."""
    E = Engine(seed)
    S = 4
    for b in range(2):
        for n in ("q_full", "q_empty", "tm_full", "tm_empty"):
            E.bar((n, b))
    for i in range(S):
        E.bar(("k_full", i)); E.bar(("k_empty", i))
    full = [Named(E, ("half_full", b)) for b in range(2)]
    empty = [Named(E, ("half_empty", b)) for b in range(2)]
    first = [sum(units[:k]) for k in range(len(units) + 1)]       # tiles before unit k
    uses = {}                                                     # (unit, tile) -> (slot, use)
    count = [0, 0]
    for k, n in enumerate(units):
        for i in range(n):
            uses[k, i] = (i & 1, count[i & 1])
            count[i & 1] += 1
    of_use = {v: t for t, v in uses.items()}

    def producer():
        for k, n in enumerate(units):
            if mistake != "q_empty":
                yield ("q_empty", k & 1), (k >> 1) - 1
            E.copies.append(("q", k, 0, [("q_full", k & 1)]))
            for i in range(n):
                t = first[k] + i
                yield ("k_empty", t % S), t // S - 1
                E.copies.append(("k", k, i, [("k_full", t % S)]))

    def mma():
        for k, n in enumerate(units):
            if mistake != "q_full":
                yield ("q_full", k & 1), k >> 1
            for i in range(n):
                t = first[k] + i
                slot, use = uses[k, i]
                yield ("k_full", t % S), t // S
                if mistake != "tm_empty":
                    yield ("tm_empty", slot), use - 1
                E.pipe.append(("mma", k, i, [("tm_full", slot), ("k_empty", t % S)]))
            E.pipe.append(("unit", k, 0, [("q_empty", k & 1)]))

    def consumer(wg):
        for k, n in enumerate(units):
            for i in range(wg, n, 2):
                slot, use = uses[k, i]
                if mistake != "tm_full":
                    yield ("tm_full", wg), use
                E.need(E.done(("mma", k, i)), "unit %d tile %d read before its MMA" % (k, i))
                E.at(("read", k, i))
                E.bars[("tm_empty", wg)].arrive()
            b = k & 1
            if wg == 1:
                if k >= 2 and mistake != "half_empty":
                    yield empty[b].arrive(wg)
                if k >= 2:
                    E.need(E.done(("half_read", k - 2)), "unit %d's statistics overwrite unit %d's" % (k, k - 2))
                E.at(("half", k))
                full[b].arrive(wg)
            else:
                at = full[b].arrive(wg)
                if mistake != "half_full":
                    yield at
                E.need(E.done(("half", k)), "unit %d's statistics read before they are written" % k)
                yield ("k_empty", 0), -1                      # the read takes a while
                E.at(("half_read", k))
                if k + 2 < len(units) and mistake != "half_empty":
                    empty[b].arrive(wg)

    def execute(kind, k, i):
        if kind == "mma":
            E.need(E.done(("q", k, 0)), "MMA of unit %d before its query rows" % k)
            E.need(E.done(("k", k, i)), "MMA of unit %d tile %d before its keys" % (k, i))
            slot, use = uses[k, i]
            if use:
                E.need(E.done(("read",) + of_use[slot, use - 1]), "MMA overwrites slot %d" % slot)
        E.at((kind, k, i))

    def land(kind, k, i):
        if kind == "q" and k >= 2:
            E.need(E.done(("unit", k - 2, 0)), "query rows of unit %d over unit %d's" % (k, k - 2))
        E.at((kind, k, i))

    return E.run({"producer": producer(), "mma": mma(), "wg0": consumer(0), "wg1": consumer(1)}, execute, land)


def run_pass2(pairs, C, layers, seed, per_layer=False, mistake=None, stray=False):
    """pairs: for each pair its segments (unit, l0, l1); every unit has `layers` layers of C chunks.

    stray adds a consumer of a pair whose share is empty and that counts itself."""
    E = Engine(seed)
    QS = 4
    parts = {}
    for segs in pairs:
        for u, l0, l1 in segs:
            parts[u] = parts.get(u, 0) + 1
    if stray:
        parts = {u: n + (1 if n > 1 else 0) for u, n in parts.items()}
    counts = {u: 0 for u in parts}
    E.bar("pass1")                                 # completion of the kernel before
    roles = {}

    def pass1():
        # an event the scheduler may delay: the counts are cleared, then the kernel ends
        yield "pass1", -1
        yield "pass1", -1
        for u in counts:
            E.need(counts[u] == 0, "unit %d counted before the counts were cleared" % u)
            counts[u] = 0
        E.at("cleared")
        E.bars["pass1"].arrive()

    def build(p, segs):
        def nm(x, i):
            return (p, x, i)
        for i in range(2):
            for x in ("k_full", "k_empty", "tm_full", "tm_empty"):
                E.bar(nm(x, i))
        for i in range(QS):
            E.bar(nm("q_full", i)); E.bar(nm("nl_full", i)); E.bar(nm("q_empty", i), 2)
        sync = Named(E, (p, "sync"))
        # the pair's chunks in order: (segment, layer, chunk) -> (qi, ki, slot, use)
        order, use, qi, ki = {}, [0, 0], 0, 0
        for s, (u, l0, l1) in enumerate(segs):
            for l in range(l0, l1):
                for c in range(C):
                    slot = (l * C + c) & 1
                    order[s, l, c] = (qi, ki, slot, use[slot])
                    use[slot] += 1
                    qi += 1
                ki += 1
        before = {(v[2], v[3]): k for k, v in order.items()}
        by_q = {v[0]: k for k, v in order.items()}

        def producer():
            waited = False
            for s, (u, l0, l1) in enumerate(segs):
                for l in range(l0, l1):
                    k = order[s, l, 0][1]
                    yield nm("k_empty", k & 1), (k >> 1) - 1
                    E.copies.append((p, "k", (s, l), [nm("k_full", k & 1)]))
                    for c in range(C):
                        q = order[s, l, c][0]
                        yield nm("q_empty", q % QS), q // QS - 1
                        E.copies.append((p, "q", (s, l, c), [nm("q_full", q % QS)]))
                        if not waited:
                            yield "pass1", 0
                            waited = True
                        E.copies.append((p, "nl", (s, l, c), [nm("nl_full", q % QS)]))

        def mma():
            for s, (u, l0, l1) in enumerate(segs):
                for l in range(l0, l1):
                    k = order[s, l, 0][1]
                    yield nm("k_full", k & 1), k >> 1
                    for c in range(C):
                        q, _, slot, n = order[s, l, c]
                        yield nm("q_full", q % QS), q // QS
                        if mistake != "tm_empty":
                            yield nm("tm_empty", slot), n - 1
                        E.pipe.append((p, "mma", (s, l, c), [nm("tm_full", slot), nm("q_empty", q % QS)]))
                    E.pipe.append((p, "layer", (s, l), [nm("k_empty", k & 1)]))

        def meet(wg):
            return sync.arrive(wg)

        def consumer(wg):
            yield "pass1", 0
            for s, (u, l0, l1) in enumerate(segs):
                buf = 0 if mistake == "red" else s & 1
                for l in range(l0, l1):
                    for c in range(C):
                        q, _, slot, n = order[s, l, c]
                        if slot != wg:
                            continue
                        yield nm("tm_full", wg), n
                        yield nm("nl_full", q % QS), q // QS
                        E.need(E.done((p, "mma", (s, l, c))), "chunk read before its MMA")
                        E.at((p, "read", (s, l, c)))
                        E.bars[nm("tm_empty", wg)].arrive()
                        E.bars[nm("q_empty", q % QS)].arrive()
                    if per_layer:
                        E.at((p, "red", buf, wg, s, l))
                        yield meet(wg)
                        if wg == 0:
                            E.need(E.done((p, "red", buf, 1, s, l)), "layer sums read before they are written")
                        yield meet(wg)
                    elif parts[u] > 1:
                        E.at(("sum", u, l, wg))
                if per_layer:
                    continue
                last = True
                if parts[u] > 1:
                    if mistake != "sums":
                        yield meet(wg)
                    if wg == 0:
                        E.need(E.done("cleared"), "unit %d counted before the counts were cleared" % u)
                        counts[u] += 1
                        E.at((p, "last", s, counts[u] == parts[u]))
                        E.at((p, "counted", s))
                    yield meet(wg)
                    E.need(E.done((p, "counted", s)), "the outcome is read before it is known")
                    last = E.done((p, "last", s, True))
                    if last:
                        for l in range(layers):
                            E.need(E.done(("sum", u, l, wg)), "unit %d layer %d added before it is there" % (u, l))
                for r in range(s):                            # the buffer's last reader is done
                    if (0 if mistake == "red" else r & 1) == buf:
                        E.need(not E.done((p, "out", r, "due")) or E.done((p, "out", r)), "sums of segment %d overwritten" % r)
                E.at((p, "red", buf, wg, s))
                if wg == 0 and last:
                    E.at((p, "out", s, "due"))
                yield meet(wg)
                if wg == 0 and last:
                    E.need(E.done((p, "red", buf, 1, s)), "sums read before they are written")
                    yield "pass1", -1                         # the read takes a while
                    E.at((p, "out", s))
                    E.at(("score", u))

        roles.update({(p, "producer"): producer(), (p, "mma"): mma(), (p, "wg0"): consumer(0), (p, "wg1"): consumer(1)})
        return order, before, by_q

    built = {p: build(p, segs) for p, segs in enumerate(pairs)}

    def execute(p, kind, at):
        if kind == "mma":
            order, before, _ = built[p]
            s, l, c = at
            _, _, slot, n = order[at]
            E.need(E.done((p, "k", (s, l))) and E.done((p, "q", at)), "MMA before its operands")
            if n:
                E.need(E.done((p, "read", before[slot, n - 1])), "MMA overwrites slot %d" % slot)
        E.at((p, kind, at))

    def land(p, kind, at):
        if kind in ("q", "nl"):
            order, _, by_q = built[p]
            q = order[at][0]
            if q >= QS:
                E.need(E.done((p, "read", by_q[q - QS])), "rows land over rows still read")
        if kind == "nl":
            E.need(E.done("cleared"), "normalisers read before pass 1 is done")
        E.at((p, kind, at))

    def empty_share(u):
        if mistake != "stray":
            yield "pass1", 0
        counts[u] += 1

    if stray:
        for u, n in parts.items():
            if n > 1:
                roles["stray", u] = empty_share(u)
    roles["pass1"] = pass1()
    got = E.run(roles, execute, land)
    if not per_layer and not stray:
        for u in parts:
            E.need(E.done(("score", u)), "unit %d has no scores" % u)
    return got


UNITS = [[], [1], [0], [2, 2, 2], [1, 1, 1, 1, 1], [3, 0, 2, 1, 0, 0, 5], [7, 4, 1, 6, 3], [0, 0, 0, 0], [12, 13, 1, 9]]


def test_pass1_sequences():
    for u in UNITS:
        for seed in range(25):
            assert run_pass1(u, seed) == "ok", u


@pytest.mark.parametrize("mistake", ["q_empty", "q_full", "tm_empty", "tm_full", "half_full", "half_empty"])
def test_pass1_planted_mistakes(mistake):
    assert _caught(lambda s: run_pass1([3, 1, 0, 0, 2, 0, 0, 5, 1, 4, 2], s, mistake)) > 0


PAIRS = [
    [[(0, 0, 7)]],                                                      # a whole unit
    [[(0, 0, 3)], [(0, 3, 7)]],                                         # one cut
    [[(0, 0, 7), (1, 0, 4)], [(1, 4, 7), (2, 0, 7), (3, 0, 3)], [(3, 3, 7)]],
    [[(0, 0, 3)], [(0, 3, 4)], [(0, 4, 7)]],                            # a share inside a unit, one layer
    [[(0, 0, 7), (1, 0, 7), (2, 0, 7), (3, 0, 4)], [], [(3, 4, 7)]],    # an empty share between two cuts
]


@pytest.mark.parametrize("per_layer", [False, True], ids=["shared", "layer"])
@pytest.mark.parametrize("C", [1, 2, 3])
@pytest.mark.parametrize("pairs", PAIRS, ids=range(len(PAIRS)))
def test_pass2_segments(pairs, C, per_layer):
    for seed in range(25):
        assert run_pass2(pairs, C, 7, seed, per_layer) == "ok"


@pytest.mark.parametrize("mistake,pairs,C,layers", [
    ("tm_empty", [[(0, 0, 7), (1, 0, 7), (2, 0, 4)], [(2, 4, 7), (3, 0, 7)]], 2, 7),
    ("red", [[(u, 0, 1) for u in range(5)]], 1, 1),                     # warpgroup 1 has no chunk and runs ahead
    ("sums", [[(0, 0, 4)], [(0, 4, 7)]], 2, 7)])
def test_pass2_planted_mistakes(mistake, pairs, C, layers):
    assert all(run_pass2(pairs, C, layers, s) == "ok" for s in range(50))
    assert _caught(lambda s: run_pass2(pairs, C, layers, s, mistake=mistake)) > 0


def test_an_empty_share_that_counts_without_waiting_is_caught():
    # with the wait it would only be a count too many, without it the count can be lost
    pairs = [[(0, 0, 3)], [(0, 3, 7)]]
    assert all(run_pass2(pairs, 2, 7, s, stray=True) == "ok" for s in range(50))
    assert _caught(lambda s: run_pass2(pairs, 2, 7, s, mistake="stray", stray=True)) > 0
