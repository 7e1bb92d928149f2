"""The signature kernel's quotient form (csrc/quotient.cuh) on the host against
Section 3.1's definition with textbook GF(2^16) products (gfpoly): the digit
recurrences as written in the source (parsed), the funnel shift of odd starts,
the remainders and the last factor of each component."""
import os
import random
import re

import pytest

from gfpoly import ginv, gmul, gpow, sig_by_polynomial

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = open(os.path.join(ROOT, "paper_2411_18183_gb300", "csrc", "quotient.cuh")).read()
M32 = 0xFFFFFFFF


def taps(name, var):
    """Offsets (ring size, [t + d, ...]) of the recurrence `name[s] = w ^ name[...] ^ ...`."""
    m = re.search(rf"{name}\[{var}\] = w\[i\] \^ ([^;]+);", SRC)
    assert m, name
    size = {"p": 16, "q": 24}[name]
    out = []
    for term in m.group(1).split("^"):
        t = re.fullmatch(rf"\s*{name}\[(?:{var}|\({var} \+ (\d+)\) % {size})\]\s*", term)
        assert t, term
        out.append(int(t.group(1) or size))
    return out


P_TAPS, Q_TAPS = taps("p", "s"), taps("q", "z")
Q_EXP = [int(x) for x in re.search(r"kQExp\[4\] = \{([^}]*)\}", SRC).group(1).split(",")]


def test_divisors_are_multiples_of_the_minimal_polynomials():
    """x^16 + ... vanishes at x, the 23rd degree one at x^3 (and so at x^6)."""
    assert sorted(P_TAPS) == [4, 13, 15, 16] and sorted(Q_TAPS) == [10, 15, 23]
    for n, tp, base in ((16, P_TAPS, 1), (23, Q_TAPS, 3)):
        v = gpow(2, base * n)
        for d in tp:
            v ^= gpow(2, base * (n - d))
        assert v == 0


def digits(words, tp):
    q = {}
    for t in range(len(words) - 1, -2, -1):               # one more step, with a zero word, at t = -1
        v = words[t] if t >= 0 else 0
        for d in tp:
            v ^= q.get(t + d, 0)
        q[t] = v
    return q


def signature(key, a):
    stream = bytes(a) + key
    stream += bytes(-len(stream) % 32)
    words = [int.from_bytes(stream[i:i + 4], "little") for i in range(0, len(stream), 4)]
    sh, sig = 8 * (a & 1), 0
    for k in (1, 2, 3, 4):
        n, tp = (23, Q_TAPS) if k == 3 else (16, P_TAPS)
        q = digits(words, tp)
        d = [((q.get(i - 1, 0) | q.get(i, 0) << 32) >> sh) & M32 for i in range(n)]
        value = 0
        for i in range(n):
            r = d[i]
            for j in (n - t for t in tp):
                if 0 < j <= i:
                    r ^= d[i - j]
            value ^= gmul(gpow(2, 2 * k * i), (r & 0xFFFF) ^ gmul(gpow(2, k), r >> 16))
        value = gmul(gmul(value, ginv(gpow(2, Q_EXP[k - 1]))), gpow(2, k * (15 - (a >> 1))))
        sig |= value << (16 * (k - 1))
    return sig


@pytest.mark.parametrize("n", [1, 2, 3, 31, 32, 33, 63, 64, 65, 127, 129, 383, 385, 700])
def test_quotient_form_gives_the_signature(n):
    rng = random.Random(n)
    for a in range(32):
        key = bytes(rng.randrange(256) for _ in range(n))
        assert signature(key, a) == sig_by_polynomial(key), (n, a)
