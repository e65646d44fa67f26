"""Roles and barriers of the tensor-memory convolution, restated on the CPU (the constants are
read from the kernel source): for every row count, dilation and segment length, in random
interleavings of the copies, the MMAs and the epilogue, every output row collects its three
input rows once and in its own accumulator block, nothing is overwritten while it is in use, and
all roles finish."""
import random
import re
from pathlib import Path

import pytest

SRC = (Path(__file__).parent.parent / "paper_2507_00294_gb300" / "csrc" / "dd_surrogate.cu").read_text()
SEG, AHEAD, SLOTS = (int(re.search(r"\b%s = (\d+)" % n, SRC).group(1)) for n in ("kSeg", "kConvAhead", "kConvMaxSlots"))


def items(H, dil, seg):
    for rho in range(dil):
        J = (H - rho + dil - 1) // dil
        for j0 in range(0, J, seg):
            j1 = min(J, j0 + seg)
            yield rho, j0, j1, J


class Bar:                       # mbarrier: wait(parity) passes once the phase of that parity is over
    def __init__(self, count):
        self.count, self.left, self.phase = count, count, 0

    def arrive(self):
        self.left -= 1
        assert self.left >= 0
        if self.left == 0:
            self.left, self.phase = self.count, self.phase + 1

    def passes(self, parity):
        return (self.phase - 1) & 1 == parity


def run(work, n_slots, rng):
    full, empty = [Bar(1) for _ in range(n_slots)], [Bar(1) for _ in range(n_slots)]
    done, free = [Bar(1) for _ in range(SEG // 2)], [Bar(1) for _ in range(SEG // 2)]
    ring, acc, got = [None] * n_slots, [None] * SEG, []

    def base_of(base, j0, j1):
        return SEG // 2 if 2 * (j1 - j0) <= SEG and base == 0 else 0

    def copies():
        n = slot = given = 0
        parity = 1
        for rho, j0, j1, J in work:
            for i in range(j0 - 1, j1 + 1, 2):
                while not empty[slot].passes(parity):
                    yield False
                assert ring[slot] is None
                ring[slot] = [(rho, r) for r in (i, i + 1) if 0 <= r <= min(j1, J - 1)]
                slot += 1
                if slot == n_slots:
                    slot, parity = 0, parity ^ 1
                n += 1
                if n > AHEAD:
                    full[given].arrive()
                    given = (given + 1) % n_slots
                yield True
        for _ in range(min(n, AHEAD)):
            full[given].arrive()
            given = (given + 1) % n_slots
        for b in range(min(n, n_slots), 0, -1):
            s = slot - b
            while not empty[s + n_slots if s < 0 else s].passes(parity if s < 0 else parity ^ 1):
                yield False

    def mmas():
        slot, base, parity, phase = 0, 0, 0, [1] * (SEG // 2)
        for rho, j0, j1, J in work:
            base = base_of(base, j0, j1)
            i0, i1 = max(j0 - 1, 0), min(j1, J - 1)
            for i in range(j0 - 1, j1 + 1, 2):
                pair = (base + i + 1 - j0) // 2
                if i + 1 < j1:
                    while not free[pair].passes(phase[pair]):
                        yield False
                    phase[pair] ^= 1
                while not full[slot].passes(parity):
                    yield False
                for ii in (i, i + 1):
                    if ii < i0 or ii > i1:
                        continue
                    assert (rho, ii) in ring[slot]
                    lo, hi = max(j0, ii - 1), min(j1 - 1, ii + 1)
                    fresh = lo if ii == i0 else ii + 1
                    assert 0 <= base + lo - j0 and base + hi - j0 < SEG and hi - lo < 3
                    for j in range(lo, hi + 1):
                        blk = base + j - j0
                        if j >= fresh:
                            assert blk // 2 == pair              # a pair this step has waited for
                            acc[blk] = (rho, j, [])
                        assert acc[blk][:2] == (rho, j) and 0 <= j - ii + 1 < 3
                        acc[blk][2].append(ii)
                yield True
                ring[slot] = None
                empty[slot].arrive()
                slot += 1
                if slot == n_slots:
                    slot, parity = 0, parity ^ 1
                if i >= j0:
                    done[pair - 1].arrive()

    def epilogue():
        base, phase = 0, [0] * (SEG // 2)
        for rho, j0, j1, J in work:
            base = base_of(base, j0, j1)
            for j in range(j0, j1, 2):
                pair = (base + j - j0) // 2
                while not done[pair].passes(phase[pair]):
                    yield False
                phase[pair] ^= 1
                for blk, jj in ((2 * pair, j), (2 * pair + 1, j + 1)):
                    if jj < j1:
                        assert acc[blk][:2] == (rho, jj)
                        got.append((rho, jj, tuple(acc[blk][2])))
                free[pair].arrive()
                yield True

    roles = [copies(), mmas(), epilogue()]
    idle = 0
    while roles:
        r = rng.choice(roles)
        try:
            idle = 0 if next(r) else idle + 1
        except StopIteration:
            roles.remove(r)
            idle = 0
        assert idle < 1000, "the roles wait on one another"
    return got


@pytest.mark.parametrize("H", [1, 2, 7, 24, 40, 128])
def test_roles(H):
    rng = random.Random(H)
    for dil in (1, 2, 3, 4, 8, 15, 16, 31, 32):
        for seg in range(3, SEG + 1):
            work = list(items(H, dil, seg))
            for cta in range(2):
                got = run(work[cta::2], rng.randint(AHEAD + 2, SLOTS), rng)
                want = [(rho, j, tuple(i for i in (j - 1, j, j + 1) if 0 <= i and rho + i * dil < H))
                        for rho, j0, j1, *_ in work[cta::2] for j in range(j0, j1)]
                assert got == want
        rows = sorted(rho + j * dil for rho, j0, j1, *_ in work for j in range(j0, j1))
        assert rows == list(range(H))
