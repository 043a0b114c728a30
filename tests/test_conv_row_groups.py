"""Host-side model of the row-by-row tcgen05 convolution's epilogue groups
(csrc/conv_tcgen05.cu): EG = 2 groups of four warps, group g % EG taking tile g, the
four warps of that group alone releasing its accumulator.  Loader, MMA issuer and the
eight epilogue warps run as coroutines in random interleavings against barriers with
the parity semantics of mbarrier waits.  Checked: a warp reads complete tiles of its
own group only, an accumulator is rewritten only after the four warps of the group
that took it have read it, the groups may run ahead of each other without a parity
wait falling two phases behind, every tile is read four times, nothing deadlocks.
A model with a wrong release count or an accumulator shared between groups fails."""
import random

import pytest

from test_conv_row_protocol import NACC, SLOTS, Bar

EG = 2


def run(items, rng, eg=EG, nacc=NACC, releases=4):
    full, aempty = [Bar(1) for _ in range(nacc)], [Bar(releases) for _ in range(nacc)]
    loaded, sfree = [Bar(1) for _ in range(SLOTS)], [Bar(1) for _ in range(SLOTS)]
    acc, tensor, copies, reads = [None] * nacc, [], [], set()

    def loader():
        for q in range(sum(n + 2 for n in items)):
            if q >= SLOTS:
                yield from sfree[q % SLOTS].wait(q // SLOTS - 1)
            copies.append(q)
            yield

    def issuer():
        q = gbase = 0
        for n in items:
            for j in range(n + 2):
                if j < n and gbase + j >= nacc:
                    yield from aempty[(gbase + j) % nacc].wait((gbase + j) // nacc - 1)
                yield from loaded[q % SLOTS].wait(q // SLOTS)
                tensor.append(("mma", [(gbase + t, j - t) for t in range(max(0, j - 2), min(n - 1, j) + 1)]))
                tensor.append(("commit", sfree[q % SLOTS]))
                if j >= 2:
                    tensor.append(("commit", full[(gbase + j - 2) % nacc]))
                q += 1
                yield
            gbase += n

    def warp(w):
        for g in range(sum(items)):
            if g % eg != w // 4:
                continue
            yield from full[g % nacc].wait(g // nacc)
            yield
            assert acc[g % nacc] == (g, 2), "a tile that is not complete or not this group's"
            reads.add((w, g))
            aempty[g % nacc].arrive()

    roles = [loader(), issuer()] + [warp(w) for w in range(4 * eg)]
    idle = 0
    while roles or tensor or copies:
        before = (len(roles), len(tensor), len(copies), len(reads), tuple(b.phase for b in loaded + sfree))
        what = rng.randrange(len(roles) + 2)
        if what < len(roles):
            try:
                next(roles[what])
            except StopIteration:
                roles.pop(what)
        elif what == len(roles) and copies:
            loaded[copies.pop(rng.randrange(len(copies))) % SLOTS].arrive()
        elif tensor:
            op = tensor.pop(0)
            if op[0] == "commit":
                op[1].arrive()
            else:
                for g, ky in op[1]:
                    a = g % nacc
                    if ky == 0 and acc[a] is not None:
                        old = acc[a][0]
                        assert all((w, old) in reads for w in range(4 * (old % eg), 4 * (old % eg) + 4)), \
                            "an accumulator rewritten before its group has read it"
                    acc[a] = (g, ky)
        after = (len(roles), len(tensor), len(copies), len(reads), tuple(b.phase for b in loaded + sfree))
        idle = idle + 1 if before == after else 0
        assert idle < 5000, "deadlock"
    assert len(reads) == 4 * sum(items)


def _items(rng):
    return [rng.choice([1, 2, 3, 7, 8, 9, 21]) for _ in range(rng.randint(1, 5))]


@pytest.mark.parametrize("seed", range(25))
def test_groups(seed):
    rng = random.Random(seed)
    run(_items(rng), rng)


@pytest.mark.parametrize("wrong", [dict(releases=8), dict(releases=3), dict(releases=2)])
def test_a_wrong_release_count_fails(wrong):
    failed = 0
    for seed in range(20):
        rng = random.Random(seed)
        try:
            run([21, 9, 21], rng, **wrong)
        except AssertionError:
            failed += 1
    assert failed == 20
