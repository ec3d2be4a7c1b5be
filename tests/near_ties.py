"""Records whose nearest centroid is decided by the rounding of the squared distances: two centroids at
nearly equal distance, kept where the rule with one rounding for the square and the sum and the rule with
two pick different clusters.  The distances are computed here in exact rationals, rounded to fp32."""
from fractions import Fraction

import numpy as np


def round32(q):
    """A rational of fp32's normal range (or zero) to the nearest fp32 value, ties to even."""
    if q == 0:
        return Fraction(0)
    a, e = abs(q), 0
    while a >= 1 << 24:
        a, e = a / 2, e + 1
    while a < 1 << 23:
        a, e = a * 2, e - 1
    m = int(a)
    rest = a - m
    m += rest > Fraction(1, 2) or (rest == Fraction(1, 2) and m % 2 == 1)
    return (1 if q > 0 else -1) * m * Fraction(2) ** e


def member(x, cent, one_rounding):
    """The assign rule on one record: features x[d], centroids cent[K][d], all fp32 values."""
    best, least = 0, None
    for k, c in enumerate(cent):
        D = Fraction(0)
        for xj, cj in zip(x, c):
            t = round32(Fraction(float(xj)) - Fraction(float(cj)))
            D = round32(t * t + D) if one_rounding else round32(round32(t * t) + D)
        if least is None or D < least:
            best, least = k, D
    return best


def likely(x, cent):
    """Whether the two rules seem to differ on x (fp64 in the place of exact arithmetic)."""
    one, two = np.zeros(len(cent), np.float32), np.zeros(len(cent), np.float32)
    for j in range(len(x)):
        t = x[j] - cent[:, j]
        one = (t.astype(np.float64) ** 2 + one).astype(np.float32)
        two = two + t * t
    return one.argmin() != two.argmin()


def records(d, K, pair, count, seed):
    """(features [count][d], centroids [K][d], memberships with one rounding): every record's membership
    is another one with two roundings.  pair: the two clusters that are near, the others lie far off."""
    rng = np.random.default_rng(seed)
    cent = (8.0 + rng.random((K, d))).astype(np.float32)
    cent[list(pair)] = rng.uniform(-1, 1, (2, d)).astype(np.float32)
    a, b = (cent[k].astype(np.float64) for k in pair)
    xs, ms = [], []
    for _ in range(100 * count):
        x = rng.uniform(-1, 1, d)
        j = int(np.argmax(np.abs(a - b)))           # this coordinate puts x where the distances are equal
        others = [i for i in range(d) if i != j]
        x[j] = (np.sum((x - a)[others] ** 2) - np.sum((x - b)[others] ** 2) + a[j] ** 2 - b[j] ** 2) / (2 * (a[j] - b[j]))
        x = x.astype(np.float32)
        if not likely(x, cent):
            continue
        m = member(x, cent, True)
        if m != member(x, cent, False):
            xs.append(x)
            ms.append(m)
            if len(xs) == count:
                return np.stack(xs), cent, np.array(ms, dtype=np.int32)
    raise AssertionError("too few records that the two rules decide differently")
