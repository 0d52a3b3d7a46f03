"""The candidate order of the tensor-core interaction (csrc/sph_interact_tc.cu,
Turns): every candidate of a piece is one column of one part, a part's columns
ascend with the candidates, the count of columns before a candidate and a hit
bit's entry offset are those of the map, and the word that ends a list leads to
the pad."""
import pytest


@pytest.mark.parametrize("turn", [False, True])
@pytest.mark.parametrize("split", [2, 4])
def test_columns_parts_and_entries_agree(split, turn):
    m, s1 = 8 // split, split - 1

    def taken(t, p):
        return p ^ ((t >> 3) & s1) if turn else p

    def entry(base, bit, p):
        e = base + 16 * split * bit
        if turn:
            e += ((bit & (m * s1)) ^ (m * p)) * (16 // m)
        return e % 2 ** 32

    for p in range(split):
        mine = [t for t in range(256) if taken(t, t & s1) == p]
        assert [t // split for t in mine] == list(range(256 // split))
        for t in range(257):
            assert sum(q < t for q in mine) == (t + s1 - taken(t, p)) // split
        for c0 in range(0, 256 // split, 8):
            base = 16 * (split * c0 + (0 if turn else p))
            for bit in range(min(32, 256 // split - c0)):
                assert entry(base, bit, p) == 16 * mine[c0 + bit]
        pad = 5000 + 16 * (1 + p if turn else split)
        assert entry(pad, 2 ** 32 - 1, p) == 5000
        if turn:
            assert {t % 8 for t in mine} == set(range(8))
