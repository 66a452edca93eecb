"""Model check, on the CPU, of how the asynchronous loops share the initializer
buffer: the count of free entries (room) that writers reserve on, with the
shortfall given back, and the order of a reader's updates.

Entry i of a buffer of C entries (stored at i mod C) has a state word, with
lap = i // C: 2 lap free for its writer, 2 lap + 1 written, 2 lap + 2 read.
Writers subtract what they want from room; those it is too few for give theirs
back; the tail moves by what is left. Then each waits for its entry to be free,
writes it and publishes it (avail). Readers claim written entries on avail,
take their indices from the head, and add them to room after that: the tail
never passes head + C, so the reader of the entry a writer waits for has claimed
it. A reader reads all it has claimed before it makes anything (a block's pass,
a warp's fill); `between` plants the mistake of reading between the steps.

Actors are generators that yield at every shared access; a seeded scheduler
interleaves them."""
import random

import pytest


class Buffer:
    def __init__(self, capacity, n_initial):
        self.C = capacity
        self.state = [0] * capacity
        self.value = [None] * capacity
        self.head, self.tail = 0, n_initial
        self.avail, self.room = n_initial, capacity - n_initial
        self.finished = 0
        for i in range(n_initial):
            self.state[i] = 1
            self.value[i] = i
        self.reads = {}
        self.live = 0
        self.errors = []

    def check(self):
        if not 0 <= self.tail - self.head <= self.C:
            self.errors.append(f"head {self.head}, tail {self.tail} of {self.C}")


def reserve(b, wants):
    """A group's lanes want wants[k] entries each; returns every lane's first
    index, or None for the lanes that wait."""
    total = sum(wants)
    got = b.room
    b.room -= total
    yield
    ends = [sum(wants[: k + 1]) for k in range(len(wants))]
    take = max([e for e in ends if e <= got], default=0)
    if take < total:
        b.room += total - take
        yield
    if take == 0:
        return [None] * len(wants)
    base = b.tail
    b.tail += take
    b.check()
    yield
    return [base + e - w if e <= take else None for e, w in zip(ends, wants)]


def write(b, index, value, bound):
    slot, lap2 = index % b.C, 2 * (index // b.C)
    for _ in range(bound):
        if b.state[slot] == lap2:
            break
        yield
    else:
        b.errors.append(f"writer of {index} waited forever")
        return
    b.value[slot] = value
    yield
    b.state[slot] = lap2 + 1
    yield
    b.avail += 1
    yield


def read(b, index, bound):
    slot, lap2 = index % b.C, 2 * (index // b.C)
    for _ in range(bound):
        if b.state[slot] == lap2 + 1:
            break
        yield
    else:
        b.errors.append(f"reader of {index} waited forever")
        return
    if index in b.reads:
        b.errors.append(f"entry {index} read twice")
    b.reads[index] = b.value[slot]
    b.live += 1
    yield
    b.state[slot] = lap2 + 2
    yield


def block(b, rng, most, made, limit, bound, between):
    tracks, unread = 0, []
    while True:
        a = b.avail
        yield
        want = min(a, rng.randint(1, most)) if a > 0 and not unread else 0
        if want > 0:
            old = b.avail
            b.avail -= want
            yield
            if old >= want:
                first = b.head
                b.head += want
                b.check()
                yield
                b.room += want
                yield
                unread = list(range(first, first + want))
            else:
                b.avail += want
                yield
        while unread:
            yield from read(b, unread.pop(0), bound)
            tracks += 1
            if between:
                break
        if not tracks:
            f = b.finished
            yield
            t = b.tail
            yield
            if f == t:
                if b.live or b.tail != b.head or b.avail:
                    b.errors.append("end concluded with work left")
                return
            continue
        # a step of a few of its tracks as one group: they end, or end and make entries
        group = min(tracks, rng.randint(1, 4))
        wants = [rng.randint(0, 2) if made[0] < limit else 0 for _ in range(group)]
        at = yield from reserve(b, wants) if sum(wants) else iter_none(group)
        ended = 0
        for w, t in zip(wants, at):
            if w == 0:
                ended += 1
            elif t is not None:
                made[0] += w
                ended += 1
                for k in range(w):
                    yield from write(b, t + k, None, bound)
        tracks -= ended
        b.live -= ended
        yield
        b.finished += ended
        if b.errors:
            return


def iter_none(n):
    yield
    return [None] * n


def run(seed, capacity, n_blocks, most, between=False, limit=60, bound=4000):
    b = Buffer(capacity, capacity // 2)
    made = [0]
    actors = [block(b, random.Random(seed * 100 + k), most, made, limit, bound, between) for k in range(n_blocks)]
    rng = random.Random(seed)
    for _ in range(3_000_000):
        if not actors or b.errors:
            return b
        actor = rng.choice(actors)
        try:
            next(actor)
        except StopIteration:
            actors.remove(actor)
    raise AssertionError("scheduler bound reached")


@pytest.mark.parametrize("capacity,most", [(4, 2), (4, 4), (8, 8), (64, 16)])
@pytest.mark.parametrize("n_blocks", [1, 2, 5])
def test_every_entry_read_once_and_room_comes_back(capacity, most, n_blocks):
    for seed in range(12):
        b = run(seed, capacity, n_blocks, most)
        assert b.errors == []
        assert sorted(b.reads) == list(range(b.tail)) and b.head == b.tail == b.finished
        assert b.avail == 0 and b.live == 0 and b.room == b.C


def test_reading_between_the_steps_is_caught():
    """A block whose claims reach around the buffer waits for itself."""
    assert any("waited forever" in e for seed in range(12) for e in run(seed, 4, 2, 4, between=True).errors)
