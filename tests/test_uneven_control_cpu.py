"""Host model of k_fft_uneven_one's hand-over between a CTA's control warp and
its compute warps, under random scheduling and partial residency.

Control, per tile: claim a ticket; look the tile up; poll its dependency; post
the tile if its inputs are there; wait for the compute warps to finish the tile
before and publish its column count; if the inputs were not there, wait for
them, then post.  Compute: take the posted tile, run it, report it done.  Every
launch must end, no row tile may run before every column tile of its chunk has
been counted, a tile's slot may not be refilled before that tile is done, and the
planted mistake -- waiting for inputs before the tile before is published --
must deadlock."""
import random

import pytest


def table(rng):
    """Tiles in ticket order: (chunk or None, is_row); a chunk's columns come
    before every row."""
    cols, rows, need = [], [], {}
    for c in range(rng.randint(1, 5)):
        n = rng.randint(1, 6)
        need[c] = n
        cols += [(c, False)] * n
        rows += [(c, True)] * rng.randint(1, 6)
    cols += [(None, False)] * rng.randint(0, 6)
    rng.shuffle(cols)
    return cols + rows, need


def run(tiles, need, ctas, resident, rng, publish_first=True):
    """True when the launch ends; asserts the orderings on the way."""
    ticket = [0]
    count = {c: 0 for c in need}
    ready = lambda t: not t[1] or count[t[0]] >= need[t[0]]

    def control(cta):
        i = 0
        while True:
            k, ticket[0] = ticket[0], ticket[0] + 1
            has = k < len(tiles)
            slot = i & 1
            if has:
                assert cta["slot"][slot] in (None, "done"), "slot refilled while in use"
                cta["slot"][slot] = tiles[k]
            posted = not has or ready(tiles[k])
            if posted:
                cta["post"].append(tiles[k] if has else None)
            if not posted and not publish_first:  # the mistake
                while not ready(tiles[k]):
                    yield
            if i > 0:
                while cta["slot"][slot ^ 1] != "done":
                    yield
                prev = cta["prev"]
                if prev[0] is not None and not prev[1]:
                    count[prev[0]] += 1
            if not posted:
                while not ready(tiles[k]):
                    yield
                cta["post"].append(tiles[k])
            if not has:
                return
            cta["prev"] = tiles[k]
            i += 1
            yield

    def compute(cta):
        i = 0
        while True:
            while not cta["post"]:
                yield
            t = cta["post"].pop(0)
            if t is None:
                return
            assert ready(t), "a row ran before its columns were counted"
            for _ in range(rng.randint(0, 3)):
                yield
            cta["slot"][i & 1] = "done"
            i += 1

    waiting = list(range(ctas))
    live = []
    idle = 0
    while waiting or live:
        while waiting and len(live) < resident:  # a CTA starts when a place is free
            waiting.pop()
            cta = {"slot": [None, None], "post": [], "prev": (None, False)}
            live.append([control(cta), compute(cta)])
        before = (ticket[0], dict(count), len(live), sum(len(w) for w in live))
        for warps in rng.sample(live, len(live)):
            for w in list(warps):
                if rng.random() < 0.7:
                    try:
                        next(w)
                    except StopIteration:
                        warps.remove(w)
        live = [w for w in live if w]
        idle = idle + 1 if before == (ticket[0], dict(count), len(live), sum(len(w) for w in live)) else 0
        if idle > 400:
            return False
    assert count == need
    return True


@pytest.mark.parametrize("seed", range(60))
def test_every_launch_ends_in_order(seed):
    rng = random.Random(seed)
    tiles, need = table(rng)
    ctas = rng.randint(1, 7)
    assert run(tiles, need, ctas, rng.randint(1, ctas), rng)


def test_waiting_before_publishing_deadlocks():
    # one CTA: its row waits for the column it has run but not yet counted
    assert not run([(0, False), (0, True)], {0: 1}, 1, 1, random.Random(1), publish_first=False)
    assert run([(0, False), (0, True)], {0: 1}, 1, 1, random.Random(1))
