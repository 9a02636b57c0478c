"""Host checks of the pruning query with classified cells: the two bits of a cell (inside: |T| < t; side:
the sign of the others) and its three parts against the settle rule, on every pattern of cells.  With f =
r/2 + 1, a coordinate is settled by n rows when at least f of their signed cells are < t and at least f
are > -t.  The functions restate k_pbits, parts 1 and 2 of k_query_bits and resolve()."""

import itertools

import numpy as np
import pytest

T1 = np.float32(1.0)
PK = int(T1.view(np.uint32))


def _bits(T):
    b = int(np.float32(T).view(np.uint32))
    return int((b & 0x7FFFFFFF) < PK), b >> 31  # inside, side


def _counts(inside, side, sign):
    """What resolve() adds to (below t, above -t) for a cell under a coordinate's sign bit."""
    below = side ^ sign
    return inside | below, inside | (below ^ 1)


def _settled(signed, f):
    return sum(v < T1 for v in signed) >= f and sum(v > -T1 for v in signed) >= f


def test_bits_count_like_the_values():
    below_t = np.nextafter(T1, np.float32(0))
    for T in [0.0, -0.0, 0.5, -0.5, below_t, -below_t, 1.0, -1.0, 2.0, -2.0, np.inf, -np.inf, 1e-45, -1e-45]:
        for sign in (0, 1):
            v = np.float32(-T if sign else T)
            assert _counts(*_bits(T), sign) == (int(v < T1), int(v > -T1)), (T, sign)


@pytest.mark.parametrize("r", [3, 4, 5, 7, 9])
def test_parts_follow_the_rule(r):
    """Part 1 settles a coordinate exactly when its first f cells do, part 2 takes those with one of the
    f outside and settles them only where f + 1 cells do; resolve() counts like the values."""
    f = r // 2 + 1
    values = [0.25, -1.0, 3.0]  # inside, outside on either side
    for cells in itertools.product(values, repeat=f + 1):
        bits = [_bits(T) for T in cells]
        none, one = 1, 1
        for inside, _ in bits[:f]:
            one = (one & inside) | none
            none &= inside
        for signs in itertools.product((0, 1), repeat=f + 1):
            signed = [np.float32(-T if s else T) for T, s in zip(cells, signs)]
            assert bool(none) == _settled(signed[:f], f)
            if one and not none:
                assert not _settled(signed[:f], f)
                if bits[f][0]:
                    assert _settled(signed, f)  # part 2; what it leaves open, part 3 decides by the signs
            counted = [_counts(i, b, s) for (i, b), s in zip(bits[:f], signs)]
            assert [sum(c) for c in zip(*counted)] == [sum(v < T1 for v in signed[:f]), sum(v > -T1 for v in signed[:f])]


def _spread(x):
    x &= 0xFFFF
    x = (x | (x << 8)) & 0x00FF00FF
    x = (x | (x << 4)) & 0x0F0F0F0F
    x = (x | (x << 2)) & 0x33333333
    return (x | (x << 1)) & 0x55555555


def test_classes_from_bits():
    """k_query_quads' classes: two bits per place out of the inside and side words, which a coordinate's sign
    swaps and one product adds to the packed counters."""
    rng = np.random.default_rng(7)
    for _ in range(200):
        inside, side = (int(v) for v in rng.integers(0, 1 << 32, 2))
        below, above = inside | side, (inside | ~side) & 0xFFFFFFFF
        words = [_spread(above) | _spread(below) << 1, _spread(above >> 16) | _spread(below >> 16) << 1]
        for n in range(32):
            cls = (words[n >> 4] >> ((n & 15) * 2)) & 3
            for sign in (0, 1):
                packed = ((cls * (0x81 if sign else 0x201)) >> (1 - sign)) & 0x101
                assert (packed & 0xFF, packed >> 8) == _counts((inside >> n) & 1, (side >> n) & 1, sign)
