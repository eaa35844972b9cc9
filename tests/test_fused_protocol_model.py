"""A host model of the two-pass persistent kernel's in-CTA barrier protocol, run
under random interleavings (no GPU).

The model follows the kernel's roles and mbarriers: the claimer's descriptor
ring and publish ring, the producer's Q buffers and K stages (one ring in tile
order, of any number of stages), one UMMA warp, each epilogue warpgroup's TMEM
buffers (tile t of a chunk belongs to warpgroup t % 2), and eight epilogue
warps with their warpgroup syncs.  Barriers keep an arrival count, a
transaction count and a phase; a wait on parity P passes when P differs from
the parity of the current phase (the PTX rule), so a waiter that falls two
phases behind -- or runs two ahead -- is misled.  TMA copies and UMMA
completions are asynchronous events.  The model checks that no barrier gets
more arrivals than its count allows, that every UMMA finds its tile and its
chunk's queries, that every epilogue warp finds its tile's logits, and that
every role finishes.
"""
import random

import pytest


class Bar:
    def __init__(self, name, count):
        self.name, self.count = name, count
        self.pending, self.tx, self.phase = count, 0, 0

    def arrive(self, tx=0):
        self.pending -= 1
        self.tx += tx
        if self.pending < 0:
            raise AssertionError(f"{self.name}: more arrivals than its count")
        self._complete()

    def land(self):
        self.tx -= 1
        if self.tx < 0:
            raise AssertionError(f"{self.name}: more bytes than expected")
        self._complete()

    def _complete(self):
        if self.pending == 0 and self.tx == 0:
            self.phase += 1
            self.pending = self.count

    def passes(self, parity):
        return parity != (self.phase & 1)


class Sim:
    """Roles (generators that yield a condition to wait for, or None) and
    timed events, interleaved at random."""

    def __init__(self, seed):
        self.rng = random.Random(seed)
        self.clock, self.events, self.order = 0, [], 0

    def at(self, time, fn):
        self.order += 1
        self.events.append((time, self.order, fn))

    def after(self, fn, lo=1, hi=30):
        self.at(self.clock + self.rng.randint(lo, hi), fn)

    def run(self, roles, limit=1_000_000):
        state = {n: None for n in roles}  # the condition each waits for
        names = sorted(roles)
        for _ in range(limit):
            if not names and not self.events:
                return
            ready = ()
            if names and (not self.events or self.rng.random() < 0.8):
                ready = (self.rng.choice(names),)
                if not self._ready(state[ready[0]]):
                    ready = () if self.events else [n for n in names if self._ready(state[n])]
                    if not ready and not self.events:
                        raise AssertionError(f"deadlock: {names}")
            if ready:
                n = self.rng.choice(ready)
                try:
                    state[n] = next(roles[n])
                except StopIteration:
                    names.remove(n)
            elif self.events and (not names or self.rng.random() < 0.5
                                  or not any(self._ready(state[n]) for n in names)):
                event = min(self.events, key=lambda e: e[:2])
                self.events.remove(event)
                self.clock = max(self.clock, event[0])
                event[2]()
        raise AssertionError("no progress (spinning roles only)")

    @staticmethod
    def _ready(condition):
        return condition is None or condition()


def _simulate(seed, stages, q_bufs, bufs_per_wg, n_chunks=30, pub=6, descs=2, forget=None):
    sim = Sim(seed)
    rng, bars = sim.rng, {}

    def mk(name, count):
        bars[name] = Bar(name, count)

    for i in range(stages):
        mk(f"full{i}", 1)
        mk(f"empty{i}", 1)
    for b in range(2 * bufs_per_wg):
        mk(f"tfull{b}", 1)
        mk(f"tempty{b}", 4)
    for i in range(descs):
        mk(f"dfull{i}", 1)
        mk(f"dempty{i}", 2 + 8)
    for i in range(q_bufs):
        mk(f"qfull{i}", 1)
        mk(f"qempty{i}", 1)
    for w in range(2):
        mk(f"wg{w}", 4)
    for i in range(pub):
        mk(f"pubfull{i}", 8)
        mk(f"pubempty{i}", 1)
    # chunks: (pass, tiles), with the short and odd-sized ones of ragged units
    chunks = [(rng.choice((1, 2)), rng.choice((1, 1, 2, 3, 5, 7, 16, 16))) for _ in range(n_chunks)]
    ring = [None] * descs
    k_stage, q_buf, tmem = [None] * stages, [None] * q_bufs, [None] * (2 * bufs_per_wg)

    def wait(name, parity):
        return lambda: bars[name].passes(parity)

    def claimer():
        issued = nxt = 0

        def pump():
            nonlocal nxt
            while nxt < issued and bars[f"pubfull{nxt % pub}"].passes((nxt // pub) & 1):
                bars[f"pubempty{nxt % pub}"].arrive()
                nxt += 1

        for c in range(n_chunks + 1):
            ds = c % descs
            while not bars[f"dempty{ds}"].passes(((c // descs) & 1) ^ 1):
                pump()
                yield None
            while issued - nxt > pub - 1:
                pump()
                yield None
            ring[ds] = None if c == n_chunks else (c, *chunks[c])
            issued += c < n_chunks
            bars[f"dfull{ds}"].arrive()
            yield None
        while nxt < issued:
            pump()
            yield None

    def producer():
        st = ph = qb = qph = 0
        for c in range(n_chunks + 1):
            ds = c % descs
            yield wait(f"dfull{ds}", (c // descs) & 1)
            d = ring[ds]
            bars[f"dempty{ds}"].arrive()
            if d is None:
                return
            yield wait(f"qempty{qb}", qph ^ 1)
            bars[f"qfull{qb}"].arrive(tx=1)

            def q_lands(q=qb, c=c):
                q_buf[q] = c
                bars[f"qfull{q}"].land()

            sim.after(q_lands)
            qb, qph = (0, qph ^ 1) if qb + 1 == q_bufs else (qb + 1, qph)
            for t in range(d[2]):
                if forget != "empty":
                    yield wait(f"empty{st}", ph ^ 1)
                bars[f"full{st}"].arrive(tx=1)

                def lands(s=st, tile=(c, t)):
                    k_stage[s] = tile
                    bars[f"full{s}"].land()

                sim.after(lands)
                st, ph = (0, ph ^ 1) if st + 1 == stages else (st + 1, ph)

    def mma():
        st = ph = qb = qph = 0
        used = [0, 0]
        busy = 0
        for c in range(n_chunks + 1):
            ds = c % descs
            yield wait(f"dfull{ds}", (c // descs) & 1)
            d = ring[ds]
            bars[f"dempty{ds}"].arrive()
            if d is None:
                return
            yield wait(f"qfull{qb}", qph)
            for t in range(d[2]):
                w = t & 1
                k = used[w]
                used[w] += 1
                b = w + 2 * (k % bufs_per_wg)
                if forget != "tempty":
                    yield wait(f"tempty{b}", ((k // bufs_per_wg) & 1) ^ 1)
                yield wait(f"full{st}", ph)
                busy = max(sim.clock, busy) + rng.randint(1, 10)

                def done(s=st, x=b, q=qb, tile=(c, t)):
                    assert k_stage[s] == tile, "another tile in the K stage"
                    assert q_buf[q] == tile[0], "another chunk's queries"
                    tmem[x] = tile
                    bars[f"tfull{x}"].arrive()
                    bars[f"empty{s}"].arrive()

                sim.at(busy, done)
                st, ph = (0, ph ^ 1) if st + 1 == stages else (st + 1, ph)
            sim.at(max(sim.clock, busy) + 1, lambda q=qb: bars[f"qempty{q}"].arrive())
            qb, qph = (0, qph ^ 1) if qb + 1 == q_bufs else (qb + 1, qph)

    def epilogue(wg):
        used = syncs = 0
        for ci in range(n_chunks + 1):
            ds = ci % descs
            yield wait(f"dfull{ds}", (ci // descs) & 1)
            d = ring[ds]
            bars[f"dempty{ds}"].arrive()
            if d is None:
                return
            for t in range(wg, d[2], 2):
                b = wg + 2 * (used % bufs_per_wg)
                yield wait(f"tfull{b}", (used // bufs_per_wg) & 1)
                used += 1
                yield None
                assert tmem[b] == (ci, t), "another tile's logits"
                bars[f"tempty{b}"].arrive()
            if d[1] == 1:  # pass 1: two warpgroup syncs
                for _ in range(2):
                    bars[f"wg{wg}"].arrive()
                    yield wait(f"wg{wg}", syncs & 1)
                    syncs += 1
            if ci >= pub:
                yield wait(f"pubempty{ci % pub}", (ci // pub - 1) & 1)
            bars[f"pubfull{ci % pub}"].arrive()

    roles = {"claimer": claimer(), "producer": producer(), "mma": mma()}
    for wg in range(2):
        for w in range(4):
            roles[f"epi{wg}.{w}"] = epilogue(wg)
    sim.run(roles)


@pytest.mark.parametrize("stages,q_bufs,bufs_per_wg", [(2, 2, 1), (3, 2, 2), (4, 2, 2), (5, 3, 4),
                                                       (4, 3, 4), (8, 3, 4), (7, 2, 1)])
def test_roles_survive_random_interleavings(stages, q_bufs, bufs_per_wg):
    for seed in range(20):
        _simulate(seed, stages, q_bufs, bufs_per_wg)


@pytest.mark.parametrize("forget", ["empty", "tempty"])
def test_a_forgotten_wait_is_caught(forget):
    """Planted in the model: the producer or the UMMA warp does not wait for
    what it overwrites."""
    for seed in range(50):
        try:
            _simulate(seed, 3, 2, 2, forget=forget)
        except AssertionError:
            return
    raise AssertionError("the forgotten wait went unnoticed")
