"""The converted sum of the fused ModUp, in exact arithmetic: its quotient comes from a sum of rounded multiply-adds, so what is left of
sum_a y_a m_a is a few times q.  The bound the device code states and the room its butterflies have are checked here for prime sets next to
2^50, where they are tightest."""
from fractions import Fraction

import numpy as np
import pytest

import fesc_synth as S

BOUND = 2.51
MAGIC = 1.5 * 2.0**52


def largest_primes(skip, count=24):
    """`count` primes = 1 mod 2^17 below 2^50 in descending order, after the first `skip`."""
    return S.ntt_primes(50, 16, skip + count, 0)[skip:]


def fma(a, b, c):
    return float(Fraction(a) * Fraction(b) + Fraction(c))


def centred(v, q):
    return v - q if v > q // 2 else v


def digit_terms(src, q):
    """m and m / q of every source limb, and the sum's starting value, as the tables hold them."""
    Q = int(np.prod([int(p) for p in src], dtype=object))
    m = [centred(Q // p % q, q) for p in src]
    mq = [float(Fraction(v, q)) for v in m]
    return m, mq, float(-(2**52) * sum(map(Fraction, mq)))


def left(y, m, mq, start, q):
    """sum y m - c q with c = the rounded quotient sum, operation by operation."""
    s = start
    for v, w in zip(y, mq):
        s = fma(2.0**52 + v, w, s)
    return sum(v * w for v, w in zip(y, m)) - int(s + MAGIC - MAGIC) * q


SETS = {"largest": largest_primes(0), "next": largest_primes(24), "shipped": S.params("full")["primes"][:24],
        "found": [1125899884167169, 1125899884036097, 1125899883642881, 1125899883380737, 1125899862016001],
        "spread": [1125899780227073, 1125899387928577, 1125899077681153, 1125899416240129, 1125899607212033]}


@pytest.mark.parametrize("name", sorted(SETS))
def test_what_is_left_of_a_converted_word(name):
    primes, g = SETS[name], np.random.default_rng(5)
    worst = 0.0
    for first in range(0, len(primes) - 1, 4):
        src = primes[first:first + 4]
        for t in [t for t in range(len(primes)) if not first <= t < first + 4][first % 3::3]:
            q = primes[t]
            m, mq, start = digit_terms(src, q)
            assert all(abs(w) <= 0.5 for w in mq)
            ys = [[0] * len(src), [p - 1 for p in src]] + [[int(g.integers(0, p)) for p in src] for _ in range(40 if len(primes) > 5 else 3000)]
            for y in ys:
                v = left(y, m, mq, start, q)
                worst = max(worst, abs(v) / q)
                assert abs(v) < 2**53                    # a signed word becomes a double in one exact conversion
    assert 0.4 < worst < BOUND, worst


@pytest.mark.parametrize("bits", [40, 45, 50])
def test_first_quotient_of_the_division_by_p(bits):
    """The fused division by P (special primes below 2^60, data primes of 2^40 to 2^50): a source word is centred, offset by 2^59 and seen by the
    FP64 sum as 2^52 plus its upper 52 bits; the quotient is in units of 2^10.  What it leaves is at most 5.2 2^10 q, which fits a signed word."""
    g = np.random.default_rng(7)
    specials = S.ntt_primes(60, 16, 4, 0)
    P = int(np.prod([int(p) for p in specials], dtype=object))
    worst = 0.0
    for q in S.ntt_primes(bits, 16, 3, 0):
        m = [centred(P // p % q, q) for p in specials]
        mq = [float(Fraction(v, 4 * q)) for v in m]
        start = float(Fraction(3, 2) * 2**52 * (1 - sum(map(Fraction, mq))))
        ys = [[0] * 4, [p - 1 for p in specials], [p // 2 for p in specials], [p // 2 + 1 for p in specials]]
        ys += [[p // 2 + (w < 0) for p, w in zip(specials, m)], [p // 2 + (w > 0) for p, w in zip(specials, m)]]      # all terms of one sign
        ys += [[int(g.integers(0, p)) for p in specials] for _ in range(2000)]
        for y in ys:
            c = [centred(v, p) for v, p in zip(y, specials)]
            s = start
            for v, w in zip(c, mq):
                s = fma(2.0**52 + ((v + 2**59) >> 8), w, s)
            assert 2.0**52 <= s < 2.0**53 and s == int(s)
            v = sum(a * b for a, b in zip(c, m)) - (int(s) - int(MAGIC)) * 2**10 * q
            worst = max(worst, abs(v) / (2**10 * q))
            assert abs(v) < 2**63
    assert worst < 5.2, worst


def stages(b, folds, count):
    """Bound (in q) after `count` stages from b: a stage takes it to 1.1875 b + 0.5, one that folds its addends first to 1 + 0.1875 b."""
    for s in range(count):
        b = 1 + 0.1875 * b if s in folds else 1.1875 * b + 0.5
        assert b < 8, (s, b)
    return b


def test_passes_whose_stages_fold_their_addends_stay_exact():
    """N = 2^16: nothing passes 8 q."""
    words = stages(1.0, {6}, 8)
    modup = stages(2 * BOUND, {1, 6}, 7)            # the first stage only adds
    moddown = stages(2 * 0.7, {5}, 7)
    assert (round(words, 2), round(modup, 2), round(moddown, 2)) == (3.38, 2.32, 3.23)
    for b in (words, modup, moddown):
        assert stages(b, {3}, 8) < 7.41 and stages(b, {3, 7}, 8) < 2.10
    product = 0.5 + 0.1875 * stages(modup, {3}, 8)  # in the key inner product
    assert 4 * product + 0.5 + 0.1875 / 2 < 8 and 4 * product + 0.5 < 8


@pytest.mark.parametrize("log_n,end", [(10, 5.88), (11, 7.48), (12, 2.41)])
def test_rounds_of_the_small_rings_stay_exact(log_n, end):
    """The seventh and the twelfth stage fold; a step's end takes the transformed word from a centred one and multiplies by a word below q
    (1/2 + 3/8 per q of the other factor), then adds a centred word of c0 and one of what the result held."""
    u = stages(1.0, {6, 11}, log_n)
    assert end - 0.02 < u < end
    assert 0.5 + u < 8 and 0.5 + 0.375 * (0.5 + u) + 0.5 + 0.5 < 8
    assert 3 * 0.875 + 0.5 < 8                     # three products of a converted word and the rest of those before


def inverse_stage(b, d):
    """Bounds of eight words after an inverse stage of distance d: sums, and products of differences with centred twiddles."""
    out = list(b)
    for i in range(8):
        if not i & d:
            out[i] = b[i] + b[i + d]
            out[i + d] = 0.5 + 0.1875 * (b[i] + b[i + d])
    assert max(out) <= 8, out
    return out


@pytest.mark.parametrize("log_n", [10, 11, 12])
def test_inverse_rounds_of_the_small_rings_stay_exact(log_n):
    """Words enter centred; log N - 9 stages, then rounds of three that fold words 0 and 4 before their last stage and 1 and 2 after it.  The words
    of a thread have one bound, as they had one place in the round before."""
    first = log_n - 9
    b = [0.5] * 8
    for s in range(first):
        b = inverse_stage(b, 1 << s)
    if first == 3:
        b[0] = b[1] = 0.5
    for last in (False, False, True):
        enter = max(b)
        assert enter <= 2
        b = inverse_stage(inverse_stage([enter] * 8, 1), 2)
        b[0] = b[4] = 0.5
        b = inverse_stage(b, 4)              # of the last round: sums and differences that the scaled products take
        if not last:
            b[1] = b[2] = 0.5
    assert 0.5 + 0.375 * max(b) < 8
