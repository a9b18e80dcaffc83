"""The digit products' arithmetic and certificate (csrc/fp64_digits.cu) in exact
integers and rationals, on the CPU: what the digits, the pairs left out and the
roundings of T and Y lose stays below the certificate's upper bound E, its lower
bound S of sum |A||X||B| holds, and so every output that it passes is within
(K + L) 2^-53 sum |A||X||B| of the exact one -- on dense, diagonal, graded and
sparse operands, on entries over 80 binary orders and on the edges of digits.

The model follows the kernel step by step (scales, balanced base-256 digits, pairs
of weight 7 at most, sums joined at 2^43, T shifted to the block's scale and cut
again); its constants are the kernel's.
"""
import math
import random
from fractions import Fraction

import pytest

LIMIT = 0.96 * 8.0  # 2^-53 in units of 2^-56, less the certificate's own roundings


def _scale(vals, least):
    """Exponent E with |v| < 2^E for all, values within 0.8 % of a power of two counted as that power; None for zeros."""
    mx = max((abs(v) for v in vals), default=0.0)
    if mx == 0:
        return None
    m, e = math.frexp(mx)
    return max(e + (1 if 2 * m >= 2 - 0x2100 / 2 ** 20 else 0), least)


def _digits(b, n):
    b = (b + 0x8080808080808080) & (2 ** 64 - 1)
    return [((b >> (56 - 8 * i)) & 255) - 128 for i in range(n)]


def _cut(x, E, n):
    """trunc(|x| 2^(63 - E)), complemented for negative x, as n balanced digits."""
    m, e = math.frexp(abs(x))
    m, s = int(m * 2 ** 53), 63 - E + e - 53
    v = m << s if s >= 0 else m >> -s
    return _digits(~v if x < 0 else v, n)


def _join(w):
    return (sum(i << (56 - 8 * s) for s, i in enumerate(w)) + (1 << 12)) >> 13


def _low(d):
    return max(abs(d) - 0.5, 0.0)


def _product(A, X, B, chunk):
    """(error, E, S, exact sum of magnitudes) of every output, in units of the product of the scales."""
    na, L, K, nb = len(A), len(A[0]), len(X), len(B)
    ea, eb = [_scale(r, -60) for r in A], [_scale(r, -60) for r in B]
    ex = _scale([v for r in X for v in r], -700)
    if ex is None:
        return []
    ek = [_scale(r, max(ex - 60, -700)) for r in X]
    zero7, zero8 = [0] * 7, [0] * 8
    da = [[_cut(v, e, 7) if e is not None else zero7 for v in r] for r, e in zip(A, ea)]
    db = [[_cut(v, e, 7) if e is not None else zero7 for v in r] for r, e in zip(B, eb)]
    dxs = [[_cut(v, e, 8) if e is not None else zero8 for v in r] for r, e in zip(X, ek)]
    hsh = 0
    while (32 << hsh) < L:
        hsh += 1
    dist = [min(ex - e, 63) if e is not None else 63 for e in ek]
    el = 0.01 + 0.033 * L + math.ceil(L / chunk) * (0.3 + 0.51 * 2 ** hsh if hsh else 0.26)
    ge = [(1.015 * sum(abs(v) for v in X[k]) * 2.0 ** -ek[k] + el) * 2.0 ** -dist[k] if ek[k] is not None else 0.0
          for k in range(K)]
    out = []
    for a in range(na):
        if ea[a] is None:
            continue
        T = []
        for k in range(K):
            t = 0
            for l0 in range(0, L, chunk):
                w = [0] * 8
                for l in range(l0, min(L, l0 + chunk)):
                    for i in range(7):
                        for j in range(8 - i):
                            w[i + j] += da[a][l][i] * dxs[k][l][j]
                assert max(abs(x) for x in w) < 2 ** 22  # whole numbers that an FP32 accumulator holds exactly
                t += _join(w) >> hsh
            T.append(t)
        m0 = max((t >> 32 if t >= 0 else ~(t >> 32)) >> min(d, 31) for t, d in zip(T, dist))
        z = 31 - (m0 + (m0 >> 7) + 1).bit_length()
        td = []
        for t, d in zip(T, dist):
            v = t << (z - d) if z >= d else t >> (d - z)
            assert 0 <= v + 0x8080808080808080 < 2 ** 64  # no carry out of the leading digit
            td.append(_digits(v, 8))
        wt = 2.0 ** (6 + hsh - z) * (sum(abs(d[0]) for d in td) * 1.02 / 128 + 0.05 * K + 0.6)
        sab = [sum(_low(da[a][l][0]) * _low(dxs[k][l][0]) for l in range(L)) * 2.0 ** -dist[k] for k in range(K)]
        for b in range(nb):
            if eb[b] is None:
                continue
            w = [0] * 8
            for k in range(K):
                for i in range(8):
                    for j in range(min(7, 8 - i)):
                        w[i + j] += td[k][i] * db[b][k][j]
            assert max(abs(x) for x in w) < 2 ** 22
            unit = Fraction(2) ** (ea[a] + ex + eb[b])
            y = _join(w) * Fraction(2) ** (6 + hsh - z - 57)
            terms = [Fraction(A[a][l]) * Fraction(X[k][l]) * Fraction(B[b][k]) / unit for k in range(K) for l in range(L)]
            E = (sum(g * (abs(d[0]) + 0.51) for g, d in zip(ge, db[b])) / 128 + wt) * 2.0 ** -56
            S = sum(s * _low(d[0]) for s, d in zip(sab, db[b])) * 2.0 ** -21
            out.append((float(abs(y - sum(terms))), E, S, float(sum(abs(t) for t in terms))))
    return out


def _operand(r, n, m):
    kind = r.choice(["dense", "diagonal", "noise", "graded", "wild", "edge"])
    if kind == "dense":
        return [[r.gauss(0, 1) for _ in range(m)] for _ in range(n)]
    if kind == "diagonal":
        return [[r.gauss(0, 1) if i == j else 0.0 for j in range(m)] for i in range(n)]
    if kind == "noise":
        return [[1.0 if i == j else 1e-9 * r.gauss(0, 1) for j in range(m)] for i in range(n)]
    if kind == "graded":
        a, b = ([10 ** (-8 * r.random()) for _ in range(k)] for k in (n, m))
        return [[r.gauss(0, 1) * a[i] * b[j] for j in range(m)] for i in range(n)]
    if kind == "wild":
        return [[0.0 if r.random() < 0.2 else r.gauss(0, 1) * 2.0 ** r.randint(-70, 10) for _ in range(m)] for _ in range(n)]
    edges = [1.0, -1.0, 1 - 2 ** -53, 2 - 2 ** -52, 1.9921875, 1.99, 0.5, -0.50390625, 2.0 ** -8, 3 * 2.0 ** -9, 0.0]
    return [[r.choice(edges) for _ in range(m)] for _ in range(n)]


@pytest.mark.parametrize("seed", range(4))
def test_errors_stay_below_the_certificate(seed):
    r = random.Random(seed)
    passed = 0
    for _ in range(150):
        K, L = r.choice([1, 2, 3, 5, 8, 16, 32]), r.choice([1, 2, 3, 5, 9, 16, 33, 70])
        ops = _operand(r, r.randint(1, 3), L), _operand(r, K, L), _operand(r, r.randint(1, 3), K)
        for err, E, S, exact in _product(*ops, r.choice([16, 32])):
            assert err <= E
            assert S <= exact * 1.025  # a digit's rest is up to 0.502 of one: within the limit's reserve
            if LIMIT * (K + L) * S * 2.0 ** -56 >= E:
                passed += 1
                assert err <= (K + L) * 2.0 ** -53 * exact
    assert passed > 150
