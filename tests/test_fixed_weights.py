"""The integer weights of the fixed-point reconstructions: each within half a unit (2^-57) of the
exact weight, the middle one within the sum of the others' roundings, and summing to 2^56."""
import os
import re
from decimal import Decimal, getcontext
from fractions import Fraction

import pytest

HEADER = os.path.join(os.path.dirname(__file__), "..", "paper_2410_05489_gb300", "csrc", "ase_df_fixed.cuh")


def nodes(n):
    getcontext().prec = 50
    s = lambda v: Decimal(v).sqrt()  # noqa: E731
    x = {1: [0], 2: [1 / s(3)], 3: [(Decimal(3) / 5).sqrt(), 0],
         4: [(Decimal(3) / 7 + 2 * s(Decimal(6) / 5) / 7).sqrt(), (Decimal(3) / 7 - 2 * s(Decimal(6) / 5) / 7).sqrt()]}[n]
    return [Fraction((1 - Decimal(v)) / 2) for v in x]  # the lower half of [0, 1], ascending


def polynomial(k):
    """Rows q: weights of W_-k .. W_k in the coefficient of xi^q (cell t is [t-1, t])."""
    n = 2 * k + 1
    A = [[(Fraction(t) ** (q + 1) - Fraction(t - 1) ** (q + 1)) / (q + 1) for q in range(n)]
         + [Fraction(int(i == j)) for j in range(n)] for i, t in enumerate(range(-k, k + 1))]
    for c in range(n):
        p = next(i for i in range(c, n) if A[i][c] != 0)
        A[c], A[p] = A[p], A[c]
        A[c] = [v / A[c][c] for v in A[c]]
        for i in range(n):
            if i != c:
                A[i] = [u - A[i][c] * v for u, v in zip(A[i], A[c])]
    return [row[n:] for row in A]


def header_rows():
    text = open(HEADER).read()
    body = text[text.index("kFixW[4] = {"):]
    body = body[:body.index("};")]
    nums = [int(v) for v in re.findall(r"-?\d+", re.sub(r"//.*", "", body[body.index("{"):]))]
    per = 9 + 9 + 4 * 10
    assert len(nums) == 4 * per
    return [nums[i * per:(i + 1) * per] for i in range(4)]


@pytest.mark.parametrize("order", [3, 5, 7, 9])
def test_weights(order):
    row = header_rows()[(order - 3) // 2]
    k = (order - 1) // 2
    P = polynomial(k)
    exact = lambda xi: [sum(xi ** q * P[q][i] for q in range(order)) for i in range(order)]  # noqa: E731
    join = lambda h, l: [(a << 28) + b for a, b in zip(h, l)]  # noqa: E731
    f = join(row[:9], row[9:18])
    assert all(abs(v) <= 1 << 27 for v in row[9:18]) and f[order:] == [0] * (9 - order)
    assert sum(f) == 1 << 56
    w = exact(Fraction(0))
    for t in range(order):
        assert abs(f[t] - w[t] * 2 ** 56) <= (Fraction(1, 2) if t != k else order)
    eh, el, oh, ol = (row[18 + 10 * i:28 + 10 * i] for i in range(4))
    G = 1 if order == 3 else k
    for g, x in enumerate(nodes(G)):
        e, o = join(eh[5 * g:5 * g + 5], el[5 * g:5 * g + 5]), join(oh[5 * g:5 * g + 5], ol[5 * g:5 * g + 5])
        assert e[0] + 2 * sum(e[1:]) == 1 << 56
        w = exact(x - 1)
        for t in range(k + 1):
            assert abs(e[t] - (w[k + t] + w[k - t]) / 2 * 2 ** 56) <= (Fraction(1, 2) if t else order)
            if t and 2 * g + 1 != G:
                assert abs(o[t] - (w[k + t] - w[k - t]) / 2 * 2 ** 56) <= Fraction(1, 2)
