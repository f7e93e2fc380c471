"""Schedule model of the convolution ring with two epilogue groups (csrc/evx_nn_tc.cu): virtual
row v belongs to group v mod 2, each group frees its rows in order, and a claim of 8 blocks
probes the last claimed row of either parity. Checked over unit sequences: a block always
belongs to the same group, the two probed rows are committed before the claiming item (no
self-wait) and imply that every claimed block is free, and a group's first stored row of a
unit is never its first row (its operands are loaded one row ahead)."""
import random

import pytest

NBLK = 16


def blk(v):
    return (NBLK - v % NBLK) % NBLK


def check(lengths):
    V, committed, vready, freed = 0, set(), NBLK - 1, {0: -2, 1: -1}  # last row known free, per group
    for L in lengths:
        for g in (0, 1):
            j0 = (g - V) & 1
            assert j0 < 2 and all((V + j) % 2 == g for j in range(j0, L + 4, 2))
        for i in range(L + 2):
            if V + i + 2 > vready:
                vc = V + i + 9
                assert vready + 8 <= vc <= vready + 10  # a new unit starts two rows further on
                for p in (vc, vc - 1):
                    assert p - NBLK in committed and blk(p) == blk(p - NBLK) and blk(p) % 2 == p % 2
                    freed[p % 2] = p - NBLK
                vready = vc
            for w in (V + i, V + i + 1, V + i + 2):
                assert w <= vready and (w < NBLK or w - NBLK <= freed[w % 2])
            committed.add(V + i)
        committed.update((V + L + 2, V + L + 3))
        V += L + 4


@pytest.mark.parametrize("lengths", [[64] * 6, [1] * 40, [2, 1, 3, 1, 2, 9, 1, 1, 30], [7, 3, 64, 2, 5, 100, 16, 15, 17]])
def test_two_groups(lengths):
    check(lengths)


def test_two_groups_random():
    rnd = random.Random(3)
    for _ in range(200):
        check([rnd.randint(1, 70) for _ in range(rnd.randint(1, 12))])
