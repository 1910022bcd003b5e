"""The tables of the two-float Gaussian start values (csrc/start_tables.cuh), recomputed in
decimal arithmetic: every entry is the pair of floats nearest to its function's value, the
second nearest to what the first leaves."""
import os
import re
from decimal import Decimal, getcontext

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HEADER = os.path.join(ROOT, "paper_2605_26261_gb300", "csrc", "start_tables.cuh")

getcontext().prec = 50
PI = Decimal("3.14159265358979323846264338327950288419716939937510")


def table(name):
    text = open(HEADER).read()
    body = re.search(name + r"\[\w+\] = \{(.*?)\n\};", text, re.S).group(1)
    rows = [[float.fromhex(v.strip().rstrip("f")) for v in row.split(",")] for row in re.findall(r"\{([^}]*)\}", body)]
    assert all(len(r) == 4 and all(float(np.float32(v)) == v for v in r) for r in rows)
    return rows


def sin_cos(a):
    s = c = Decimal(0)
    term = Decimal(1)
    for k in range(60):
        if k % 2:
            s += term if k % 4 == 1 else -term
        else:
            c += term if k % 4 == 0 else -term
        term = term * a / (k + 1)
    return s, c


def check(hi, lo, value):
    rest = value - Decimal(hi)
    assert abs(rest) <= Decimal(float(np.spacing(np.float32(abs(hi))))) / 2, (hi, value)
    assert abs(rest - Decimal(lo)) <= Decimal(float(np.spacing(np.float32(abs(lo))))) / 2, (lo, rest)


def test_log_table():
    rows = table("kLogTable")
    assert len(rows) == 182
    for i, (rh, rl, lh, ll) in enumerate(rows):
        check(rh, rl, Decimal(2) ** -23 / (181 + i))
        check(lh, ll, (Decimal(181 + i) / 256).ln())


def test_trig_table():
    rows = table("kTrigTable")
    assert len(rows) == 129
    for i, (sh, sl, ch, cl) in enumerate(rows):
        s, c = sin_cos(PI * i / 512)
        check(sh, sl, s)
        check(ch, cl, c)
