"""Host-side model of the row-by-row tcgen05 convolution's barriers
(csrc/conv_tcgen05.cu): loader, MMA issuer and epilogue as coroutines in random
interleavings, barriers with the parity semantics of mbarrier waits.  Checked:
every MMA reads the row it expects, each accumulator receives its three rows in
order ky = 0, 1, 2 and is initialised first, no copy lands in a slot that an
unfinished MMA reads, no accumulator is rewritten before its epilogue has read
it, no parity wait falls two phases behind, and nothing deadlocks."""
import random

import pytest

SLOTS, NACC = 8, 8


class Bar:
    def __init__(self, count):
        self.count = self.pending = count
        self.phase = 0

    def arrive(self):
        self.pending -= 1
        if self.pending == 0:
            self.pending, self.phase = self.count, self.phase + 1

    def wait(self, k):  # the wait for completed phase k, as a parity wait sees it
        while not (self.phase > 0 and ((self.phase - 1) & 1) == (k & 1)):
            assert self.phase <= k, "a parity wait fell two phases behind"
            yield
        assert self.phase == k + 1


def run(items, rng):
    full, aempty = [Bar(1) for _ in range(NACC)], [Bar(4) for _ in range(NACC)]
    loaded, sfree = [Bar(1) for _ in range(SLOTS)], [Bar(1) for _ in range(SLOTS)]
    slot_row, acc = [None] * SLOTS, [None] * NACC
    copies, tensor, done = [], [], []

    def loader():
        q = 0
        for n in items:
            for _ in range(n + 2):
                if q >= SLOTS:
                    yield from sfree[q % SLOTS].wait(q // SLOTS - 1)
                copies.append(q)
                q += 1
                yield

    def issuer():
        q = gbase = 0
        for n in items:
            for j in range(n + 2):
                lo, hi = max(0, j - 2), min(n - 1, j)
                if j < n and gbase + j >= NACC:
                    yield from aempty[(gbase + j) % NACC].wait((gbase + j) // NACC - 1)
                yield from loaded[q % SLOTS].wait(q // SLOTS)
                tensor.append(("mma", q, [(gbase + t, j - t) for t in range(lo, hi + 1)]))
                tensor.append(("commit", sfree[q % SLOTS]))
                if j >= 2:
                    tensor.append(("commit", full[(gbase + j - 2) % NACC]))
                q += 1
                yield
            gbase += n

    def warp(w):
        for g in range(sum(items)):
            yield from full[g % NACC].wait(g // NACC)
            assert acc[g % NACC] == (g, 2)
            yield
            done.append((w, g))
            aempty[g % NACC].arrive()

    roles = [loader(), issuer()] + [warp(w) for w in range(4)]
    idle = 0
    while roles or tensor or copies:
        what = rng.randrange(len(roles) + 2)
        before = (len(roles), len(tensor), len(copies), len(done), tuple(b.phase for b in loaded + sfree))
        if what < len(roles):
            try:
                next(roles[what])
            except StopIteration:
                roles.pop(what)
        elif what == len(roles) and copies:
            q = copies.pop(rng.randrange(len(copies)))
            assert not any(op[0] == "mma" and op[1] % SLOTS == q % SLOTS for op in tensor), "copy into a slot in use"
            slot_row[q % SLOTS] = q
            loaded[q % SLOTS].arrive()
        elif tensor:
            op = tensor.pop(0)
            if op[0] == "commit":
                op[1].arrive()
            else:
                assert slot_row[op[1] % SLOTS] == op[1]
                for g, ky in op[2]:
                    a = g % NACC
                    if ky == 0:
                        assert acc[a] is None or all((w, acc[a][0]) in done for w in range(4))
                    else:
                        assert acc[a] == (g, ky - 1)
                    acc[a] = (g, ky)
        after = (len(roles), len(tensor), len(copies), len(done), tuple(b.phase for b in loaded + sfree))
        idle = idle + 1 if before == after else 0
        assert idle < 5000, "deadlock"
    assert len(done) == 4 * sum(items)


@pytest.mark.parametrize("seed", range(25))
def test_rows(seed):
    rng = random.Random(seed)
    run([rng.choice([1, 2, 3, 7, 8, 9, 21]) for _ in range(rng.randint(1, 5))], rng)
