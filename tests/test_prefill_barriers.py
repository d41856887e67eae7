"""The order of the chunk prefill's named barriers, on a model of its warps: random schedules, and waits that run out anywhere.

A named barrier counts arrivals.  A warp that is there twice before the others have been there once completes it too early, and from then
on somebody waits without end.  The order must therefore not hang on anybody's speed, least of all on how long a wait that has run out
looked on."""
import os
import random
import re

import pytest

SOURCE = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2510_09608_b200", "csrc", "svlm_prefill_sm100.cu")

# what the model below goes through, role by role and in the order of the source: operation, barrier, tile (g: its own, o: the other one), threads
ISSUER = ["sync READ o 160", "arrive ASKED - 64", "sync META - 128", "sync Q g 160", "sync P1 g 160", "sync P2 g 160", "arrive PV g 160", "sync READ 1 160"]
RELAY = ["sync META - 128", "arrive S 0 160", "arrive S 1 160", "sync ASKED - 64", "arrive S g 160"]
SOFTMAX = ["sync S g 160", "arrive Q g 160", "sync Q g 160", "sync S g 160", "sync PV g 160"]
PAGE = ["arrive READ g 160", "sync PV g 160", "sync PV g 160", "arrive P1 g 160", "arrive P2 g 160"]


def test_the_model_is_of_the_source():
    src = re.sub(r"//(?! =====)[^\n]*", "", open(SOURCE).read())
    tile = {"": "0", "g": "g", "(g ^ 1)": "o", "1": "1"}

    def ops(begin, end):
        part = src[src.index(begin):]
        found = re.findall(r"bar_(sync|arrive)\(BAR_(\w+)(?: \+ ([^,]+))?, (\d+)\)", part[:part.index(end)])
        return [f"{op} {name} {'-' if name in ('META', 'ASKED') else tile[at]} {n}" for op, name, at, n in found if name != "WG"]
    assert ops("= MMA issuer of tile g", "= warp 11") == ISSUER
    assert ops("= warp 11", "= softmax warpgroups") == RELAY
    assert ops("= softmax warpgroups", "if (sh.abort_flag)") == SOFTMAX
    assert ops("void softmax_page", "struct PfPages") == PAGE


class _Barrier:
    def __init__(self):
        self.gen, self.there, self.need = 0, set(), None

    def arrive(self, who, threads):
        assert who not in self.there, ("twice in one generation", who)
        assert self.need in (None, threads), ("two sizes in one generation", who)
        self.need = threads
        self.there.add(who)
        if 32 * len(self.there) == threads:
            self.gen, self.there, self.need = self.gen + 1, set(), None


def _run(seed, segs, p_out):
    """segs: pages of the thread block's units; p_out: how likely a wait runs out at a look."""
    rnd = random.Random(seed)
    bars = {(b, g): _Barrier() for b in ("READ", "S", "Q", "P1", "P2", "PV") for g in (0, 1)}
    bars["META"] = bars["ASKED"] = _Barrier()        # one of the hardware's
    queue, done, gave_up = [], set(), [False]        # products asked for, one issuer's in order; those that are through
    loaded, stored = {}, {}                          # pages whose S all four warps have taken, whose P they have put down

    def sync(b, who, threads):
        gen = bars[b].gen
        bars[b].arrive(who, threads)
        while bars[b].gen == gen:
            yield

    def wait(what):                                  # on an mbarrier: True, or it runs out
        while rnd.random() >= (p_out if not gave_up[0] else max(p_out, 0.3)):
            if what is None or what in done:
                return True
            yield
        gave_up[0] = True
        return False

    def producer():                                  # (the ring's own mbarriers: always possible, or they run out as the issuers' waits do)
        yield from sync("META", "tma", 128)

    def issuer(g):
        me, ok, steps, pvs = ("issuer", g), True, 0, 0
        yield from sync("META", me, 128)

        def step():
            nonlocal steps
            if g == 1 or steps > 0:
                yield from sync(("READ", g ^ 1), me, 160)
            if ok:
                before = ("S", g ^ 1, steps if g else steps - 1)
                assert gave_up[0] or before[2] < 0 or loaded.get(before) == 4, "scores overwritten"
                queue.append(("S", g, steps))
            steps += 1
            bars["ASKED"].arrive(me, 64)
        for n in segs:
            if n and ok:
                ok = yield from wait(None)
            yield from sync(("Q", g), me, 160)
            if n:
                yield from step()
            for j in range(n):
                if ok:
                    ok = yield from wait(None)
                if j + 1 < n:
                    yield from step()
                yield from sync(("P1", g), me, 160)
                yield from sync(("P2", g), me, 160)
                if ok:
                    assert gave_up[0] or stored.get((g, pvs)) == 4, "weights not there"
                    queue.append(("PV", g, pvs))
                    ok = yield from wait(("PV", g, pvs))
                bars["PV", g].arrive(me, 160)
                pvs += 1
        if g == 0 and steps:
            yield from sync(("READ", 1), me, 160)

    def relay():
        ok, steps = True, 0
        yield from sync("META", "relay", 128)
        for g in (0, 1):
            bars["S", g].arrive("relay", 160)
        for n in segs:
            for _ in range(n):
                for g in (0, 1):
                    if ok:
                        ok = yield from wait(("S", g, steps))
                    yield from sync("ASKED", "relay", 64)
                    bars["S", g].arrive("relay", 160)
                steps += 1

    def softmax(g, w):
        me, page = ("softmax", g, w), 0
        yield from sync(("S", g), me, 160)
        for n in segs:
            if n:
                bars["Q", g].arrive(me, 160)
            else:
                yield from sync(("Q", g), me, 160)
            for j in range(n):
                yield from sync(("S", g), me, 160)
                assert gave_up[0] or ("S", g, page) in done, "scores not there"
                loaded["S", g, page] = loaded.get(("S", g, page), 0) + 1
                bars["READ", g].arrive(me, 160)
                yield
                if j:
                    yield from sync(("PV", g), me, 160)
                    assert gave_up[0] or ("PV", g, page - 1) in done, "weights overwritten"
                stored[g, page] = stored.get((g, page), 0) + 1
                bars["P1", g].arrive(me, 160)
                yield
                bars["P2", g].arrive(me, 160)
                yield
                page += 1
            if n:
                yield from sync(("PV", g), me, 160)
    warps = [producer(), relay(), *(issuer(g) for g in (0, 1)), *(softmax(g, w) for g in (0, 1) for w in range(4))]
    for _ in range(60000):
        if not warps:
            break
        k = rnd.randrange(len(warps))
        try:
            for _ in range(rnd.choice((1, 1, 2, 10))):
                next(warps[k])
        except StopIteration:
            del warps[k]
        if queue and rnd.random() < 0.5:
            g = rnd.choice(queue)[1]
            first = next(x for x in queue if x[1] == g)
            queue.remove(first)
            done.add(first)
    assert not warps, "somebody waits without end"
    assert not any(b.there for b in bars.values())


@pytest.mark.parametrize("p_out", [0.0, 0.005, 0.1, 1.0])
def test_named_barriers_keep_their_order(p_out):
    for seed in range(150):
        rnd = random.Random(seed)
        _run(seed, [rnd.choice((0, 1, 1, 2, 3, 5)) for _ in range(rnd.randint(1, 4))], p_out)
