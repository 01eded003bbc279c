"""The quotient of two bf16 values as csrc/quantize_w4.cu forms it - q = x r with r = 1 / s, then q + (x - q s) r, every operation
rounded to 32 bits - is the correctly rounded one: all pairs of 8-bit mantissas, in exact arithmetic (signs and exponents only scale)."""
from fractions import Fraction as Fr


def rn(v):
    """A positive or negative fraction (or zero) rounded to 24 significant bits, ties to even."""
    if v == 0:
        return Fr(0)
    f, e = abs(v), 0
    while f >= 2:
        f, e = f / 2, e + 1
    while f < 1:
        f, e = f * 2, e - 1
    n, r = divmod(f * 2 ** 23, 1)
    if r > Fr(1, 2) or (r == Fr(1, 2) and n % 2):
        n += 1
    return (1 if v > 0 else -1) * n * Fr(2) ** (e - 23)


def test_all_pairs_of_mantissas():
    for s in range(128, 256):
        r = rn(Fr(1, s))
        for x in range(128, 256):
            q = rn(x * r)
            left = x - q * s
            assert rn(left) == left  # the remainder is exact
            assert rn(q + left * r) == rn(Fr(x, s)), (x, s)
