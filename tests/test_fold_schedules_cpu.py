"""The compiled schedules of the folded passes are those of one rule."""
import os
import re

from paper_2005_00322_gb300 import build

OPS = {1: 0, 2: 4, 3: 16, 4: 16, 5: 40, 8: 52}      # real operations of a butterfly


def ops(n):
    if n in OPS:
        return OPS[n]
    p = next(q for q in (4, 2, 3, 5) if n % q == 0)
    h = n // p
    return p * ops(h) + h * ops(p) + 4 * (p - 1) * (h - 1)


def lanes(R, A, B):
    return max((R // 2 + 1) * max(A, B), A * B // 2 + 1)


def cost(R, A, B):
    NR, nk = R // 2 + 1, A * B // 2 + 1
    p1, p2, p3 = ops(A) + 10 * A, ops(B) + 10 * B, 2 * ops(R) + 20 * R
    c = 0.33 * lanes(R, A, B) * (2 * p1 + 2 * p2 + p3) + 0.67 * (2 * NR * B * p1 + 2 * NR * A * p2 + nk * p3)
    if R > 10:
        c *= 1.1
    for limit in (10, 16):
        if max(R, A, B) > limit:
            c *= 1.2
    return c


def by_rule(L):
    inner = [1, 2, 3, 4, 5, 6, 8, 9, 10, 12, 15, 16]
    every = [(R, A, L // R // A) for R in range(2, 21, 2) if L % R == 0 for A in inner
             if L // R % A == 0 and L // R // A in inner]
    if any(s[0] < 10 and lanes(*s) <= 48 for s in every):
        every = [s for s in every if s[0] != 10]
    R, A, B = min(every, key=lambda s: cost(*s))
    n = lanes(R, A, B)
    return R, A, B, 8 if n <= 48 else 4, 8 if n <= 20 else 4 if n < 60 else 2


def test_every_entry_is_the_rules():
    src = open(os.path.join(build.CSRC, "pstd_fold_list.h")).read()
    table = {}
    for e in re.findall(r"X\((\d+), (\d+), (\d+), (\d+), (\d+)\)", src):
        R, A, B, PS, PC = map(int, e)
        assert R * A * B not in table
        table[R * A * B] = (R, A, B, PS, PC)

    def smooth(n):
        for q in (2, 3, 5):
            while n % q == 0:
                n //= q
        return n == 1
    assert set(table) == {2 * n for n in range(24, 1025) if smooth(n) and n not in (25, 625)}
    # between equal costs the order of the two inner radices is free
    for L, e in table.items():
        r = by_rule(L)
        assert e == r or (e[0] == r[0] and {e[1], e[2]} == {r[1], r[2]} and e[3:] == r[3:] and cost(*e[:3]) == cost(*r[:3])), (L, e, r)
