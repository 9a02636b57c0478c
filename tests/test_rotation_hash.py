"""Host check of the query's hash arithmetic: a hash value x held as Y = 8 (x + 1), reduced by the
carry-out of a 64-bit addition.  The functions restate rot_add, rot_mul and rot_at with Python
integers, word by word; they are compared with the definition at the extremes of every operand, at
the sums that just reach p, and on random operands."""

import numpy as np

P61 = (1 << 61) - 1
M32, M64 = (1 << 32) - 1, (1 << 64) - 1


def _rot_add(y, s8):
    total = y + s8
    carry = total >> 64
    return ((total & M64) + 8 * carry) & M64


def _rot_mul(a8, i):
    w = (a8 & M32) * i
    z = (a8 >> 32) * i + (w >> 32)
    assert w <= M64 and z <= M64
    return _rot_add((z & M32) << 32 | (w & M32), 8 * (z >> 32) + 8)


def test_bucket_of_any_column_count():
    """x mod c by the 64-bit inverse floor(2^64 / c): the quotient's estimate is at most 1 too small for
    every x < 2^61, so the low words alone give the remainder."""
    rng = np.random.default_rng(3)
    cs = [3, 5, 6, 7, 777, 30_011, (1 << 26) - 1, (1 << 25) + 1] + [int(v) for v in rng.integers(3, 1 << 26, 50)]
    for c in (c for c in cs if c & (c - 1)):
        inv = M64 // c
        xs = [0, 1, c - 1, c, c + 1, P61 - 1, P61 - 2, (P61 - 1) // c * c, (P61 - 1) // c * c - 1]
        for x in xs + [int(v) % P61 for v in rng.integers(0, 1 << 62, 200)]:
            r = ((x & M32) - ((x * inv >> 64) & M32) * c) & M32
            assert (r - c if r >= c else r) == x % c


def _rep(x):
    return 8 * (x + 1)


def test_addition_reduces_exactly():
    xs = [0, 1, 2, 7, P61 - 1, P61 - 2, P61 // 2, P61 // 2 + 1, 1 << 60]
    rng = np.random.default_rng(1)
    xs += [int(v) % P61 for v in rng.integers(0, 1 << 62, 200)]
    for x in xs:
        for s in xs + [P61 - x - 1, (P61 - x) % P61, (P61 - x + 1) % P61]:
            assert _rot_add(_rep(x), 8 * s) == _rep((x + s) % P61)


def test_hash_matches_the_definition():
    rng = np.random.default_rng(2)
    a_s = [1, 2, P61 - 1, P61 - 2, 1 << 60, (1 << 32) - 1, 1 << 32] + [int(v) % (P61 - 1) + 1 for v in rng.integers(0, 1 << 62, 40)]
    b_s = [0, 1, P61 - 1] + [int(v) % P61 for v in rng.integers(0, 1 << 62, 5)]
    i_s = [0, 1, 2, 3, (1 << 31) - 2, (1 << 31) - 1, (1 << 31) + 127] + [int(v) for v in rng.integers(0, 1 << 31, 40)]
    for a in a_s:
        for i in i_s:
            assert _rot_mul(8 * a, i) == _rep(a * i % P61)
            for b in b_s + [(-a * i) % P61]:
                y = _rot_add(_rot_mul(8 * a, i), 8 * b)
                x = (a * i + b) % P61
                assert y == _rep(x)
                for c in (1, 64, 1 << 18, 1 << 26):
                    assert (((y & M32) >> 3) - 1) % c == x % c      # bucket
                    assert ((y & M32) >> 3) % c == (x + 1) % c      # place
                assert ((~y & 8) >> 3) == x & 1                     # sign bit
                for t in (1, 2, 3):                                 # the other coordinates of a quad
                    assert _rot_add(y, 8 * (t * a % P61)) == _rep((a * (i + t) + b) % P61)
