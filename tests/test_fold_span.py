"""Slots that a single row launch writes (span_slots), restated on the CPU:
for every row tile, the ranks of the blocks whose items meet it (span_slot)
must be exactly 0 .. span_slots - 1, so that the fold of unzeroed slots reads
every written slot and no other."""
import random

import pytest


def span_slots(n, tiles, sc, x):
    t = tiles * sc
    k_lo = ((x * sc + 1) * n - 1) // t
    k_hi = ((x + 1) * sc * n - 1) // t
    return k_hi - k_lo + 1


def written(n, tiles, sc):
    """Ranks written per tile by the blocks' segments."""
    t = tiles * sc
    out = [[] for _ in range(tiles)]
    for k in range(n):
        f, hi = t * k // n, t * (k + 1) // n
        while f < hi:
            x = f // sc
            out[x].append(k - ((x * sc + 1) * n - 1) // t)
            f = min(hi, (x + 1) * sc)
    return out


def cases():
    rng = random.Random(5)
    fixed = [(152, 2, 4096), (152, 512, 4), (152, 512, 1), (1, 64, 3), (152, 152, 1), (151, 2, 76), (304, 16, 1000)]
    return fixed + [(0, 1 << rng.randint(0, 9), rng.randint(1, 300)) for _ in range(40)]


@pytest.mark.parametrize("nb,tiles,sc", cases())
def test_written_ranks_are_the_slots_the_fold_reads(nb, tiles, sc):
    n = min(nb or 152, tiles * sc)
    for x, ranks in enumerate(written(n, tiles, sc)):
        assert ranks == list(range(span_slots(n, tiles, sc, x)))
        assert len(ranks) <= n // tiles + 2


@pytest.mark.parametrize("n2", [2, 4, 8])
def test_short_fold_reads_and_writes_name_the_same_channel_once(n2):
    """reduce2048_short_kernel: row position 128 q1 + 8 q2 + q3 holds k1 = q1 + 16 q2 + 256 q3."""
    seen = [0] * (2048 * n2)
    for b in range(64 * n2):
        q2 = b // (4 * n2)
        reads = {}
        for e in range(32):
            m, q3 = 4 * (b % (4 * n2)) + (e >> 3), e & 7
            reads[e] = (m % n2, 128 * (m // n2) + 8 * q2 + q3)
        for e in range(32):
            k2, pos = reads[8 * (e & 3) + (e >> 2)]
            k = 4 * (b % (4 * n2)) + (e & 3) + 16 * n2 * q2 + 256 * n2 * (e >> 2)
            q1, p2, q3 = pos // 128, pos // 8 % 16, pos % 8
            assert k == k2 + n2 * (q1 + 16 * p2 + 256 * q3)
            seen[k] += 1
    assert seen == [1] * (2048 * n2)
