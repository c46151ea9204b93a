"""The multiplication that replaces division by the grid sizes: exact for every
0 <= n < 2^31 (floor(n m / 2^(31+k)), 2^k >= d, m = ceil(2^(31+k) / d) < 2^32)."""
import pytest


def fast_div(d):
    k = 0
    while (1 << k) < d:
        k += 1
    return ((1 << (31 + k)) + d - 1) // d, 31 + k


@pytest.mark.parametrize("d", [1, 2, 3, 5, 7, 31, 32, 33, 251, 255, 256, 257, 384, 1000, 4095, 32767, 65535, 16776960])
def test_division_by_multiplication_is_exact(d):
    m, shift = fast_div(d)
    assert m < 1 << 32
    top = (1 << 31) - 1
    for q in {0, 1, 2, top // d - 1, top // d, top // (2 * d)}:
        for n in (q * d - 1, q * d, q * d + 1, q * d + d - 1, top):
            if 0 <= n <= top:
                assert (n * m) >> shift == n // d
                assert n * m < 1 << 64
