"""The tensor-core base conversion's epilogue in exact integers: lo + t with
t = 2^16 hi - floor(hi floor(2^48 / p) / 2^32) p and no reduction between stays below 2^32 for
every prime below 2^31, is congruent to lo + 2^16 hi, and is below 2 p for primes above the
kernel's limit (read from its source), so that one conditional subtraction completes it."""
import os
import random
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2512_18345_gb300", "csrc",
                   "bconv_tc.cu")
TOP = (1 << 30) + (1 << 22)  # lo, hi of a 12-input contraction are below this
LIMIT = int(re.search(r"kBigPrime = (\d+)u;", open(SRC).read()).group(1))


@pytest.mark.parametrize("p", [2 ** 20 + 7, 2 ** 29 + 11, 2 ** 30 - 35, LIMIT - 1, LIMIT + 1, 3 * 2 ** 29, 2 ** 31 - 1])
def test_epilogue(p):
    g = random.Random(p)
    w16s = (65536 << 32) // p
    div32 = (1 << 32) // p
    # the values whose quotient estimate falls furthest short: 2^16 hi just below a multiple of p
    his = [TOP - 1, 0, 1] + [g.randrange(TOP) for _ in range(2000)]
    his += [min(TOP - 1, (k * p - 1) >> 16) for k in (1, 2, (TOP << 16) // p - 1, (TOP << 16) // p)]
    for hi in his:
        t = (hi * 65536 - ((hi * w16s) >> 32) * p) % (1 << 32)
        assert t == hi * 65536 - ((hi * w16s) >> 32) * p and t < 1.251 * p
        for lo in (0, TOP - 1, g.randrange(TOP)):
            v = lo + t
            assert v < 1 << 32
            if p > LIMIT:
                assert v < 2 * p
            else:
                v = v - ((v * div32) >> 32) * p
                assert 0 <= v < 2 * p
            assert v % p == (lo + 65536 * hi) % p
