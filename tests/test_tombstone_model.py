"""Model of batched inserts and erases with threads interleaved at every
memory access (no GPU): claims that reuse tombstones, and erases that leave an
EMPTY slot where no probe chain passes.

Each thread is a generator that yields between its accesses; a random
scheduler picks who goes next.  Checked after every batch, from tables with
long runs of full buckets and tombstones: no key in two slots, the expected
key set, the probe-chain invariant (every key is found), under the preferred-
slot protocol its invariant, and the used-slot count that the claims and
erases keep.  The kernels are checked against the oracle by the GPU tests."""
import random

import pytest

EMPTY, TOMB = "E", "T"


class Table:
    """Slots hold EMPTY, TOMB, ("key", k), ("claim", k) or ("mark", k)."""

    def __init__(self, n_buckets, S, spread):
        self.nb, self.S, self.spread = n_buckets, S, spread
        self.slots = [EMPTY] * (n_buckets * S)
        self.used = 0

    def home(self, k):  # spread < nb crowds the keys into a few buckets
        return ((k * 2654435761 + 97) % (1 << 32) >> 8) % self.spread

    def pref(self, k):
        return ((k * 2246822519 + 13) % (1 << 32) >> 5) % self.S

    def bucket(self, b):
        return range(b * self.S, (b + 1) * self.S)

    def find(self, k):
        b = self.home(k)
        for _ in range(self.nb):
            words = [self.slots[i] for i in self.bucket(b)]
            if ("key", k) in words:
                return True
            if EMPTY in words:
                return False
            b = (b + 1) % self.nb
        return False

    def cas(self, i, old, new):
        seen = self.slots[i]
        if seen == old:
            self.slots[i] = new
        return seen

    # ---- insert: one thread per key (equal keys allowed)
    def claim(self, k, pref_first):
        mine, same = ("claim", k), (("claim", k), ("key", k))
        if pref_first:  # blind CAS of the preferred slot
            yield
            seen = self.cas(self.home(k) * self.S + self.pref(k), EMPTY, mine)
            if seen == EMPTY or seen in same:
                return
        yield
        words = [self.slots[i] for i in self.bucket(self.home(k))]  # one bucket load
        if any(w in same for w in words):
            return
        if EMPTY in words:
            i = self.home(k) * self.S + self._pick(k, words, pref_first)
            yield
            if self.cas(i, EMPTY, mine) == EMPTY:
                return
        yield from self._walk(k, pref_first)

    def _pick(self, k, words, pref_first):
        p = self.pref(k)
        return p if pref_first and words[p] == EMPTY else words.index(EMPTY)

    def _walk(self, k, pref_first):
        mine, same = ("claim", k), (("claim", k), ("key", k))
        while True:
            b, tomb, lost = self.home(k), None, False
            for probe in range(self.nb):
                yield
                words = [self.slots[i] for i in self.bucket(b)]
                if any(w in same for w in words):
                    return
                if EMPTY not in words:
                    if tomb is None and TOMB in words:
                        tomb = b * self.S + words.index(TOMB)
                    b = (b + 1) % self.nb
                    if probe + 1 < self.nb or tomb is None:
                        continue
                i, free = (tomb, TOMB) if tomb is not None else (
                    b * self.S + self._pick(k, words, pref_first and probe == 0), EMPTY)
                yield
                seen = self.cas(i, free, mine)
                if seen == free:
                    self.used -= free == TOMB
                    return
                if seen in same:
                    return
                lost = True
                break
            assert lost, "the table is full"

    # ---- erase: one thread per marked slot
    def resolve(self, i, pref_placed):
        b = i // self.S
        yield
        words = [self.slots[j] for j in self.bucket(b)]
        live = [w[1] for w in words if w[0] == "key"]
        preferred = pref_placed and any(self.pref(k) == i % self.S for k in live)
        to_empty = EMPTY in words
        if not to_empty and not preferred:
            nb = (b + 1) % self.nb
            empty, displaced = False, nb == b
            for j in self.bucket(nb):
                yield
                w = self.slots[j]
                empty |= w == EMPTY
                displaced |= w[0] == "key" and self.home(w[1]) != nb
            to_empty = empty and not displaced
        yield
        self.slots[i] = EMPTY if to_empty and not preferred else TOMB
        self.used -= self.slots[i] == EMPTY


def run_all(rnd, threads):
    threads = list(threads)
    while threads:
        t = rnd.choice(threads)
        try:
            next(t)
        except StopIteration:
            threads.remove(t)


@pytest.mark.parametrize("pref_first", [False, True])
@pytest.mark.parametrize("S,n_buckets,spread", [(4, 12, 12), (4, 12, 3), (4, 1, 1), (8, 6, 2), (4, 30, 20)])
@pytest.mark.parametrize("seed", range(8))
def test_interleaved_batches_keep_the_table(pref_first, S, n_buckets, spread, seed):
    rnd = random.Random(seed * 1009 + n_buckets * 7 + S + pref_first)
    t = Table(n_buckets, S, spread)
    live = set()
    room = int(0.7 * len(t.slots))
    universe = range(4 * len(t.slots))
    for _ in range(120):
        if rnd.random() < 0.5:
            fresh = rnd.sample(universe, rnd.randint(1, max(1, room // 2)))
            fresh = [k for k in fresh if k in live or len(live | {k}) <= room]
            room_left = max(0, room - len(live))
            new = [k for k in fresh if k not in live][:room_left]
            old = [k for k in fresh if k in live]
            batch = new + old + [rnd.choice(new + old) for _ in range(len(new))] if new + old else []
            run_all(rnd, [t.claim(k, pref_first) for k in batch])
            claimed = [w[1] for w in t.slots if w[0] == "claim"]
            assert len(claimed) == len(set(claimed)), "equal keys took two slots"
            assert set(claimed) == set(new)
            t.slots = [("key", w[1]) if w[0] == "claim" else w for w in t.slots]
            t.used += len(claimed)
            live |= set(new)
        elif live:
            out = rnd.sample(sorted(live), rnd.randint(1, len(live)))
            marked = [i for i, w in enumerate(t.slots) if w[0] == "key" and w[1] in out]
            for i in marked:
                t.slots[i] = ("mark", t.slots[i][1])
            run_all(rnd, [t.resolve(i, pref_first) for i in marked])
            live -= set(out)
        stored = [w[1] for w in t.slots if w[0] == "key"]
        assert len(stored) == len(set(stored)) and set(stored) == live
        assert all(t.find(k) for k in live), "probe chain broken"
        assert t.used == sum(w != EMPTY for w in t.slots)
        if pref_first:
            for k in live:
                assert t.slots[t.home(k) * t.S + t.pref(k)] != EMPTY, "preferred-slot invariant broken"


def test_a_sliding_window_does_not_lengthen_the_runs():
    """Batches that come and go over a fixed set: with tombstones reused and
    chains closed, the table keeps EMPTY slots in nearly every bucket."""
    rnd = random.Random(1)
    t = Table(400, 4, 400)
    run_all(rnd, [t.claim(k, False) for k in range(500)])
    t.slots = [("key", w[1]) if w[0] == "claim" else w for w in t.slots]
    full = []
    for r in range(60):
        batch = [10_000 + (r % 4) * 1_000 + j for j in range(130)]
        run_all(rnd, [t.claim(k, False) for k in batch])
        t.slots = [("mark", w[1]) if w[0] == "claim" else w for w in t.slots]
        run_all(rnd, [t.resolve(i, False) for i, w in enumerate(t.slots) if w[0] == "mark"])
        full.append(sum(all(t.slots[i] != EMPTY for i in t.bucket(b)) for b in range(t.nb)))
    assert max(full[30:]) <= max(full[:10]) + 4
