"""The tables of the FP64 draws' functions (usp_math64.cuh) against 40-digit
arithmetic: the logarithm's reciprocals and logarithms, and the sines and
cosines with their low parts."""
import math
import os
import re

import pytest

from paper_1808_03801_gb300 import build

mp = pytest.importorskip("mpmath")
FOLD = 106


def _table(name):
    with open(os.path.join(build.CSRC, "usp_math64.cuh")) as f:
        text = f.read()
    body = text[text.index(f"{name}[256] = {{"):]
    body = body[:body.index("};")]
    pairs = re.findall(r"\{(-?[0-9a-fx.p+-]+), (-?[0-9a-fx.p+-]+)\}", body)
    assert len(pairs) == 256
    return [tuple(float.fromhex(v) if "x" in v else float(v) for v in p) for p in pairs]


def test_logarithm_table():
    with mp.workdps(40):
        for i, (inv, log) in enumerate(_table("kLogTab")):
            half = 0.5 if i >= FOLD else 1.0
            lo, hi = half * (1 + i / 256), half * (1 + (i + 1) / 256)
            assert (math.frexp(inv)[0] * 2 ** 21).is_integer()   # 20 fraction bits
            # the remainder z inv - 1 of an argument of the interval: an interval's width on either side at most
            assert max(abs(lo * inv - 1), abs(hi * inv - 1)) <= 1 / 256, i
            ref = -mp.log(mp.mpf(inv))
            assert abs(mp.mpf(log) - ref) <= 0.003 * math.ulp(abs(log)) if log else ref == 0, i


def test_turn_tables():
    with mp.workdps(40):
        for k, ((s, c), (ls, lc)) in enumerate(zip(_table("kTurnTab"), _table("kTurnLow"))):
            a = 2 * mp.pi * k / 256
            # exact at the quarters, where mpmath's own argument is rounded
            sin, cos = ((0, 1), (1, 0), (0, -1), (-1, 0))[k // 64] if k % 64 == 0 else (mp.sin(a), mp.cos(a))
            for hi, low, ref in ((s, ls, sin), (c, lc, cos)):
                assert abs(mp.mpf(hi) - ref) <= 0.5 * math.ulp(hi), k
                assert abs(mp.mpf(hi) + mp.mpf(low) - ref) <= math.ulp(abs(low)) if low else hi == ref, k
