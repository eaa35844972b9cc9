"""A host model of the resident kernel's protocols, run under random
interleavings (no GPU).

`_simulate` has several CTAs with the kernel's roles: descriptors, TMA, UMMA,
two warpgroups of four warps, the sums, the two denominator warps and the
announcements; mbarriers and asynchronous completions are those of
test_fused_protocol_model.py.  Tensor memory is a ring of 512 columns and of 16
tiles, a unit's sums are a count that every CTA adds its chunks to, and some
units take the second round (own chunk sums read back, a ticket that all
chunks must add to).  The model checks that what a role reads is what was
written for it (K stages, query buffers, tensor-memory tiles before and after
pass 1, denominators, chunk sums), that no barrier gets more arrivals than its
count, that no columns are written while they hold logits that are still to be
read, and that the call completes.

`_start` models the start of the call: which CTAs take part, and as what.
"""
import random

import pytest

from test_fused_protocol_model import Bar, Sim

DESCS, TILES, PUB, COLUMNS, GRID, PAIRS = 32, 16, 8, 512, 152, 20
P1, P2 = 1, 2


def _units(rng, rows, ct, most_chunks, n):
    out = []
    for _ in range(n):
        nch = rng.choice((1, 1, 2, 3, rng.randint(1, most_chunks), most_chunks))
        out.append({"nch": nch, "last": rng.randint(1, ct), "width": rng.choice(rows), "ct": ct,
                    "slow": rng.random() < 0.2})
    return out


def _simulate(seed, grid, rows, ct, stages, q_bufs, lse=False, apart=False, n_units=8,
              most_chunks=None, ring=None, hold=None):
    sim = Sim(seed)
    rng = sim.rng
    hold = hold or COLUMNS // (ct * max(rows))  # chunks of a unit in tensor memory
    units = _units(rng, rows, ct, most_chunks or (3 if apart else 1) * grid * hold, n_units)
    ring = ring or PAIRS * GRID // grid
    chunks = [(u, cc) for u, U in enumerate(units) for cc in range(U["nch"])]
    first = [sum(V["nch"] for V in units[:u]) for u in range(n_units)]
    summed, ticket, scored = [0] * n_units, [0] * n_units, [0] * n_units
    roles = {}

    def cta(me):
        bars = {}

        def mk(name, count):
            bars[name] = Bar(f"cta{me}.{name}", count)

        for i in range(stages):
            mk(f"full{i}", 1)
            mk(f"empty{i}", 1)
        for i in range(TILES):
            mk(f"tfull0.{i}", 1)
            mk(f"tfull1.{i}", 1)
            mk(f"tempty{i}", 4)
        for i in range(DESCS):
            mk(f"dfull{i}", 1)
            mk(f"dempty{i}", 14)
        for i in range(q_bufs):
            mk(f"qfull{i}", 1)
            mk(f"qempty{i}", 1)
        for i in range(2):
            mk(f"p1full{i}", 4)
            mk(f"p1empty{i}", 1)
            for k in range(2):
                mk(f"dnfull{i}.{k}", 1)
                mk(f"dnempty{i}.{k}", 4)
        for i in range(PUB):
            mk(f"p2full{i}", 4)
            mk(f"p2empty{i}", 1)
        descs = [None] * DESCS
        k_stage, q_buf, tmem = [None] * stages, [None] * q_bufs, [None] * TILES
        live = {}  # tile slot -> columns, from its UMMA to its last read
        dens, sums, pairs = {}, [None, None], [None] * ring
        sum_pos, p2_unit = [0], [None] * PUB

        def wait(name, parity):
            return lambda: bars[name].passes(parity)

        def scheduler():
            mine = [x for x in range(len(chunks)) if x % grid == me]
            if apart:  # a unit's pass 1, then pass 2 of the one before
                runs = {}
                for x in mine:
                    runs.setdefault(chunks[x][0], []).append(x)
                order, prev = [], None
                for u in [*runs, None]:
                    if u is not None:
                        order += [(x, P1) for x in runs[u]]
                    if prev is not None:
                        order += [(x, P2) for x in runs[prev]]
                    prev = u
            else:
                order = [(x, P2 if lse else P1 | P2) for x in mine]
            end = tile = 0
            last, den_unit = None, None
            for c, (x, mode) in enumerate([*order, (None, 0)]):
                ds = c % DESCS
                yield wait(f"dempty{ds}", ((c // DESCS) & 1) ^ 1)
                if x is None:
                    descs[ds] = {"mode": 0}
                else:
                    u, cc = chunks[x]
                    U = units[u]
                    nt = U["last"] if cc == U["nch"] - 1 else ct
                    full = ct * U["width"]
                    col = (end + full - 1) // full * full
                    if col + full > COLUMNS:
                        col = 0
                    end = col + full
                    den_unit = den_unit if mode == P1 else u
                    descs[ds] = {
                        "mode": mode, "wg": c & 1 if lse else 1, "new_q": (u, mode) != last,
                        "last_q": x + grid >= first[u] + U["nch"], "u": u, "den": den_unit, "x": x,
                        "x_last": x + (first[u] + U["nch"] - 1 - x) // grid * grid, "nt": nt,
                        "col": col, "width": U["width"], "tile": tile}
                    last = (u, mode)
                    tile += nt
                bars[f"dfull{ds}"].arrive()

        def each():
            """(condition, None, None) to wait for, then (None, descriptor,
            its slot), for every chunk of this CTA and the end."""
            c = 0
            while True:
                ds = c % DESCS
                yield wait(f"dfull{ds}", (c // DESCS) & 1), None, None
                d = descs[ds]
                yield None, d, ds
                if d["mode"] == 0:
                    return
                c += 1

        def producer():
            st = ph = qb = qph = 0
            for cond, d, ds in each():
                if d is None:
                    yield cond
                    continue
                if d["mode"] == 0:
                    return
                if d["new_q"]:
                    yield wait(f"qempty{qb}", qph ^ 1)
                    bars[f"qfull{qb}"].arrive(tx=1)

                    def q_lands(q=qb, u=d["u"]):
                        q_buf[q] = u
                        bars[f"qfull{q}"].land()

                    sim.after(q_lands)
                    qb, qph = (0, qph ^ 1) if qb + 1 == q_bufs else (qb + 1, qph)
                d = dict(d)
                bars[f"dempty{ds}"].arrive()
                for t in range(d["nt"]):
                    yield wait(f"empty{st}", ph ^ 1)
                    bars[f"full{st}"].arrive(tx=1)

                    def lands(s=st, what=(d["x"], t)):
                        k_stage[s] = what
                        bars[f"full{s}"].land()

                    sim.after(lands)
                    st, ph = (0, ph ^ 1) if st + 1 == stages else (st + 1, ph)

        def mma():
            st = ph = 0
            qb, nq, qph = 0, 0, 0
            tile = oldest = end = busy = 0
            at = {}
            for cond, d, ds in each():
                if d is None:
                    yield cond
                    continue
                d = dict(d)
                bars[f"dempty{ds}"].arrive()
                if d["mode"] == 0:
                    return
                if d["new_q"]:
                    qb = nq
                    yield wait(f"qfull{qb}", qph)
                    nq, qph = (0, qph ^ 1) if nq + 1 == q_bufs else (nq + 1, qph)
                col = d["col"]
                for t in range(d["nt"]):
                    wrap = col < end
                    while oldest < tile:
                        c0, c1 = at[oldest % TILES]
                        over = c0 < col + d["width"]
                        if not (tile - oldest >= TILES or ((c1 > end or over) if wrap
                                                           else (c1 > end and over))):
                            break
                        yield wait(f"tempty{oldest % TILES}", (oldest // TILES) & 1)
                        oldest += 1
                    yield wait(f"full{st}", ph)
                    b = tile % TILES
                    at[b] = (col, col + d["width"])
                    for o, (c0, c1) in live.items():
                        assert c1 <= col or col + d["width"] <= c0, "columns still to be read"
                    live[b] = at[b]
                    busy = max(sim.clock, busy) + rng.randint(1, 10)

                    def done(s=st, b=b, q=qb, what=(d["x"], t), u=d["u"],
                             w=0 if d["mode"] & P1 else d["wg"]):
                        assert k_stage[s] == what, "another tile in the K stage"
                        assert q_buf[q] == u, "another unit's queries"
                        tmem[b] = what
                        bars[f"tfull{w}.{b}"].arrive()
                        bars[f"empty{s}"].arrive()

                    sim.at(busy, done)
                    st, ph = (0, ph ^ 1) if st + 1 == stages else (st + 1, ph)
                    tile += 1
                    end = col + d["width"]
                    col += d["width"]
                if d["last_q"]:
                    sim.at(max(sim.clock, busy) + 1, lambda q=qb: bars[f"qempty{q}"].arrive())

        def freed(tile):
            b = tile % TILES
            last = bars[f"tempty{b}"].pending == 1
            if last:
                live.pop(b)
            bars[f"tempty{b}"].arrive()

        def pass1(w):
            k1 = tile = 0
            ph = 0
            for cond, d, ds in each():
                if d is None:
                    yield cond
                    continue
                if d["mode"] == 0:
                    return
                if d["mode"] & P1:
                    b = k1 & 1
                    yield wait(f"p1empty{b}", ((k1 >> 1) & 1) ^ 1)
                    for t in range(d["nt"]):
                        s = (tile + t) % TILES
                        yield wait(f"tfull0.{s}", (ph >> s) & 1)
                        ph ^= 1 << s
                        assert tmem[s] == (d["x"], t), "another tile's logits (pass 1)"
                    sums[b] = d["x"]
                    bars[f"p1full{b}"].arrive()
                    k1 += 1
                tile += d["nt"]
                bars[f"dempty{ds}"].arrive()

        def sum_role():
            k1 = 0
            for cond, d, ds in each():
                if d is None:
                    yield cond
                    continue
                if d["mode"] == 0:
                    return
                if d["mode"] & P1:
                    b = k1 & 1
                    yield wait(f"p1full{b}", (k1 >> 1) & 1)
                    assert sums[b] == d["x"], "another chunk's sums"
                    summed[d["u"]] += 1
                    pairs[k1 % ring] = d["x"]
                    yield None
                    bars[f"p1empty{b}"].arrive()
                    sum_pos[0] = d["x"] + 1
                    k1 += 1
                    if d["mode"] == P1:
                        for t in range(4 * d["nt"]):
                            freed(d["tile"] + (t >> 2))
                bars[f"dempty{ds}"].arrive()

        def pass2(wg, w):
            k2 = tile = ph = 0
            unit, kd = None, -1
            for cond, d, ds in each():
                if d is None:
                    yield cond
                    continue
                if d["mode"] == 0:
                    return
                if d["mode"] & P2:
                    if d["wg"] == wg:
                        if d["den"] != unit:
                            if kd >= 0:
                                bars[f"dnempty{wg}.{kd & 1}"].arrive()
                            kd += 1
                            yield wait(f"dnfull{wg}.{kd & 1}", (kd >> 1) & 1)
                            unit = d["den"]
                        for t in range(d["nt"]):
                            s = (tile + t) % TILES
                            if d["mode"] == P2:
                                yield wait(f"tfull{wg}.{s}", (ph >> s) & 1)
                                ph ^= 1 << s
                            yield None
                            assert dens[wg, kd & 1] == d["u"], "another unit's denominators"
                            assert tmem[s] == (d["x"], t), "another tile's logits (pass 2)"
                            freed(tile + t)
                        yield wait(f"p2empty{k2 % PUB}", ((k2 // PUB) & 1) ^ 1)
                        p2_unit[k2 % PUB] = unit
                        bars[f"p2full{k2 % PUB}"].arrive()
                    k2 += 1
                tile += d["nt"]
                bars[f"dempty{ds}"].arrive()

        def announce():
            nxt = 0
            for cond, d, ds in each():
                if d is None:
                    yield cond
                    continue
                if d["mode"] == 0:
                    return
                bars[f"dempty{ds}"].arrive()
                if d["mode"] & P2:
                    yield wait(f"p2full{nxt % PUB}", (nxt // PUB) & 1)
                    scored[p2_unit[nxt % PUB]] += 1
                    bars[f"p2empty{nxt % PUB}"].arrive()
                    nxt += 1

        def denominators(mine):
            unit, k = [None, None], [0, 0]
            for cond, d, ds in each():
                if d is None:
                    yield cond
                    continue
                if d["mode"] == 0:
                    return
                w = d["wg"]
                if d["den"] != unit[w]:
                    kw = k[w]
                    k[w] += 1
                    unit[w] = d["den"]
                    if kw & 1 == mine:
                        u, d0 = d["den"], d
                        yield wait(f"dnempty{w}.{mine}", ((kw >> 1) & 1) ^ 1)
                        if not lse:
                            yield lambda: summed[u] == units[u]["nch"]
                            if units[u]["slow"]:
                                yield lambda: sum_pos[0] > d0["x_last"]
                                own = range(d0["x"], d0["x_last"] + 1, grid)
                                for x in own:
                                    assert pairs[x // grid % ring] == x, "another chunk's pairs"
                                ticket[u] += len(own)
                                yield lambda: ticket[u] == units[u]["nch"]
                                for x in own:
                                    assert pairs[x // grid % ring] == x, "another chunk's pairs"
                        dens[w, mine] = u
                        bars[f"dnfull{w}.{mine}"].arrive()
                bars[f"dempty{ds}"].arrive()

        roles[f"{me}.sched"] = scheduler()
        roles[f"{me}.tma"] = producer()
        roles[f"{me}.mma"] = mma()
        roles[f"{me}.sum"] = sum_role()
        roles[f"{me}.ann"] = announce()
        for m in range(2):
            roles[f"{me}.den{m}"] = denominators(m)
        for w in range(4):
            roles[f"{me}.wg0.{w}"] = pass2(0, w) if lse else pass1(w)
            roles[f"{me}.wg1.{w}"] = pass2(1, w)

    for me in range(grid):
        cta(me)
    sim.run(roles)
    assert scored == [U["nch"] for U in units]


@pytest.mark.parametrize("grid,rows,ct,stages,q_bufs,kw", [
    (3, (32,), 4, 4, 3, {}),              # four chunks of four tiles
    (3, (32, 64), 4, 4, 3, {}),           # two
    (4, (32, 64), 2, 5, 3, {}),
    (2, (64, 96, 128), 2, 3, 2, {}),
    (3, (64, 128, 192), 1, 2, 2, {}),
    (1, (32, 64), 1, 4, 3, {}),
    (3, (32,), 1, 8, 3, {"ring": PAIRS, "n_units": 14}),  # the ring of chunk sums of a full grid
    (3, (32, 64), 4, 4, 3, {"lse": True}),
    (2, (64, 192), 1, 2, 2, {"lse": True}),
    (3, (32, 64), 4, 4, 3, {"apart": True}),  # more chunks than tensor memory holds
    (2, (64, 128, 192), 1, 2, 2, {"apart": True}),
    (1, (32,), 2, 4, 3, {"apart": True}),
])
def test_roles_survive_random_interleavings(grid, rows, ct, stages, q_bufs, kw):
    for seed in range(6):
        _simulate(seed, grid, rows, ct, stages, q_bufs, **kw)


@pytest.mark.parametrize("kw", [
    {"most_chunks": 9},  # a unit of more chunks than the CTAs hold, both passes at once: they wait for ever
    {"ring": 1, "n_units": 14},  # chunk sums overwritten before the second round has read them
])
def test_a_mistake_is_caught(kw):
    for seed in range(40):
        try:
            _simulate(seed, 2, (64,), 4, 4, 3, **kw)
        except AssertionError:
            return
    raise AssertionError("the mistake went unnoticed")


# ------------------------------------------------------------------ the start
CLOSED, APART = 1 << 31, 1 << 30


def _start(seed, n, held, stale=False):
    """n CTAs of which the last `held` start only when an earlier one has left;
    every atomic operation is one step.  Returns what each became.  stale: the
    words hold anything at first."""
    rng = random.Random(seed)
    word = {"arrive": 0, "past": 0, "zeroed": 0, "slots": 0}
    if stale:
        word = {"arrive": rng.choice((rng.getrandbits(32), rng.randrange(2 * n),
                                      CLOSED | rng.getrandbits(18))),
                "past": rng.getrandbits(32), "zeroed": rng.getrandbits(32),
                "slots": rng.choice((rng.getrandbits(n), (1 << n) - 1))}
    sms = list(range(n))
    rng.shuffle(sms)
    out = {}
    patience = rng.choice((3, 30, 300))  # polls before a CTA gives up on the others
    apart_after = rng.choice((1, 10, 1000))

    def cta(block):
        old = word["arrive"]
        word["arrive"] = (old + 1) % 2**32
        me, grid, w, polls = block, n, (old + 1) % 2**32, 0
        yield
        while w != n:
            if w & CLOSED:
                me = None if old & CLOSED else old & 0xFFFF
                grid = (w >> 16) & 0x3FFF
                break
            count = w & 0xFFFF
            if count == n:
                slot = sms[block] if rng.random() < 0.9 else rng.randrange(n)  # may have changed
                me = None
                for _ in range(n):
                    yield
                    if not word["slots"] >> slot & 1:
                        word["slots"] |= 1 << slot
                        me = slot
                        break
                    slot = (slot + 1) % n
                break
            polls += 1
            if polls > patience:
                if word["arrive"] == w:
                    word["arrive"] = CLOSED | count << 16 | count
            elif polls > apart_after and not w & APART:
                if word["arrive"] == w:
                    word["arrive"] = w | APART
            yield
            w = word["arrive"]
            yield
        if me is not None and (me >= grid or grid > n):
            me = None
        out[block] = (me, grid)
        if me is not None:
            word["zeroed"] += 1
            yield
            polls = 0
            while word["zeroed"] < grid and not (stale and polls > 300):  # the wait runs out
                polls += 1
                yield
        word["past"] += 1
        if word["past"] == n:
            word.update(arrive=0, past=0, zeroed=0, slots=0)

    waiting = [cta(b) for b in range(n)]
    running = [waiting.pop(0) for _ in range(n - held)]
    for _ in range(400_000):
        if not running:
            break
        r = rng.choice(running)
        try:
            next(r)
        except StopIteration:
            running.remove(r)
            if waiting:  # its SM is free
                running.append(waiting.pop(0))
    assert not running and not waiting, "the start does not end"
    assert stale or not any(word.values()), "the words are not ready for the next call"
    return out


@pytest.mark.parametrize("n,held", [(1, 0), (2, 0), (7, 0), (7, 1), (7, 6), (40, 11)])
def test_the_ctas_agree_on_who_takes_part(n, held):
    for seed in range(150):
        out = _start(seed, n, held)
        assert len(out) == n
        parts = sorted(me for me, _ in out.values() if me is not None)
        assert parts == list(range(len(parts))) and parts
        assert {grid for _, grid in out.values()} == {len(parts)}
        assert len(parts) <= n - held or not held


@pytest.mark.parametrize("n", [1, 2, 7, 40, 152])
def test_a_start_on_stale_words_ends_within_bounds(n):
    """A workspace that was never initialised: no number beyond the grid (the
    CTAs index their scratch by it), and no CTA that stays."""
    for seed in range(100):
        for me, grid in _start(seed, n, 0, stale=True).values():
            assert me is None or 0 <= me < grid <= n
