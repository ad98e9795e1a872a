"""CPU: the hash tables of the sparse input, level by level, transcribed from the
device routines (slot of a key at a level, linear probing, the table's size).  A
level past its capacity keeps the entries it reads first, those at the front of
the table; their children must spread over the whole of the next table, or the
probes become as long as the table."""
import numpy as np
import pytest

U = np.uint64


def first_slots(keys, beta, slots):
    k = keys.astype(U) ^ U(beta * 0x9e3779b9 & 0xffffffff)
    k ^= k >> U(16)
    k = k * U(0x7feb352d) & U(0xffffffff)
    k ^= k >> U(15)
    k = k * U(0x846ca68b) & U(0xffffffff)
    k ^= k >> U(16)
    return (k * U(slots) >> U(32)).astype(np.int64)


def fill(keys, beta, slots):
    """The table's keys in its order, and the mean number of probes."""
    table = np.full(slots, -1, dtype=np.int64)
    probes = 0
    for key, at in zip(keys.tolist(), first_slots(keys, beta, slots).tolist()):
        probes += 1
        while table[at] >= 0:
            probes += 1
            at = 0 if at + 1 == slots else at + 1
        table[at] = key
    return table[table >= 0], probes / len(keys)


def children(keys, n, beta):
    rb, cb = keys >> (n + beta) & 1, keys >> beta & 1
    kI = keys & ~((1 << beta) | (1 << (n + beta)))
    kX, kY = kI | 1 << beta, kI | 1 << (n + beta)
    diag = rb == cb
    return np.unique(np.concatenate([np.where(diag, kI, kX), np.where(diag, kX | kY, kY)]))


@pytest.mark.parametrize("n,m,cap", [(10, 100, 1424), (10, 100, 5000), (12, 300, 1500), (14, 50, 2000)])
def test_entries_kept_past_the_capacity_spread_over_the_next_table(n, m, cap):
    g = np.random.default_rng(n)
    keys = np.unique(g.integers(0, 2 ** n, m) << n | g.integers(0, 2 ** n, m))
    slots, passed = 2 * cap + cap // 2, 0
    for beta in range(n):
        keys, probes = fill(children(keys, n, beta), beta, slots)
        assert probes <= 8                                   # load 0.8: 3 expected
        passed += len(keys) > cap
        keys = keys[:cap]
    assert passed >= 2
