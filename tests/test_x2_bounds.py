"""Bounds of the FP64-accurate product's digits and of its level sums, from digits made with test_x2_digits' restatement of the
kernel.  A float pair in the top binades meets the largest fourth digit (128 of the first number and 64 of the
second's integer part), one whose last place is half a fourth digit's unit the largest fifth.  From the bounds: the
sums of 128 columns at levels 0-5 are at most 2^24, integers that FP32 holds whatever the order; level 6 can
pass 2^24, where each of its (at most 56) additions may lose one unit, of weight 2^-48."""
import numpy as np
from test_x2_digits import F, digits

BOUND = [128, 128, 128, 192, 192, 128, 128]


def test_digit_bounds():
    rng = np.random.default_rng(9)
    most = np.zeros(7)
    for e in range(7, -40, -1):  # binades of the scaled entry, up to 2^7
        n = 20000
        man = rng.integers(2 ** 23, 2 ** 24, n).astype(np.float64)
        # remainders of every size, and just short of half a unit; bit patterns that round up all the way
        man[:2000] = 2 ** 24 - 1 - rng.integers(0, 64, 2000)
        man[2000:4000] = 2 ** 23 + rng.integers(0, 64, 2000) * 2 ** rng.integers(0, 17, 2000)
        hi = (man * 2.0 ** (e - 24)).astype(F) * rng.choice(np.array([-1, 1], F), n)
        half = 2.0 ** (e - 25) * rng.choice([-1.0, 1.0], n)
        lo = (half * np.where(np.arange(n) % 2, 1 - 2.0 ** -20, rng.uniform(0, 1, n))).astype(F)
        most = np.maximum(most, np.abs(digits(hi, lo, 0)).max(1))
    assert np.all(most <= BOUND), most
    assert most[3] > 160 and most[4] > 160, most  # the two wider bounds are needed


def test_level_sums():
    for level in range(7):
        s = 128 * sum(BOUND[i] * BOUND[level - i] for i in range(level + 1))
        assert s <= 2 ** 24 if level < 6 else 2 ** 24 < s < 2 ** 25
    # level 6: 56 additions (8 steps x 7 products) of a unit, against the largest entries' product (2^12 or more)
    assert 56 * 2.0 ** -48 <= 2.0 ** -54 * 2 ** 12
    # what is left out of one term: digit products of i + j >= 7 and the tails (half a unit of the seventh digit times
    # an entry, twice), against the same product
    tail = sum(BOUND[i] * BOUND[7 - i] for i in range(1, 7)) * 2.0 ** -56 * 1.01 + 2 * 2.0 ** 7 * 2.0 ** -49
    assert tail <= 2.0 ** -50 * 2 ** 12
