"""The stated rounding of the wavenumber sweep's chunk map, in NumPy FP32 (a fused
multiply-add formed in FP64, which holds the product of two FP32 numbers
exactly): the rule for the rows left over, read from the source, is that of
groups of four, two and one rows, and the fused chain is as close to the exact
map as the unfused one."""
import os
import re

import numpy as np
import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1812_05711_gb300", "csrc")
f = np.float32


def _tail_rule():
    text = open(os.path.join(SRC, "sweep_dev.cuh")).read()
    rule = re.search(r"constexpr bool tail_row_fused\(int i, int rem\) \{ return (.*?); \}", text).group(1)
    rule = rule.replace("||", " or ").replace("&&", " and ")
    return lambda i, rem: bool(eval(rule, {"i": i, "rem": rem}))


def _fused(n):
    tail, rem = _tail_rule(), n % 8
    return [i > 0 for _ in range(n // 8) for i in range(8)] + [tail(i, rem) for i in range(rem)]


def test_rows_left_over_are_groups_of_four_two_and_one():
    for rem in range(8):
        groups = [i > 0 for size in (4, 2, 1) if rem & size for i in range(size)]
        assert _fused(rem) == groups, rem


def _map(r, d, fused):
    br, df, rp = f(0), f(0), f(0)
    for k in range(len(r)):
        df = f(float(d[k]) - float(rp) * float(df)) if fused[k] else f(d[k] - br)
        br = f(r[k] * df)
        rp = r[k]
    return br


@pytest.mark.parametrize("n", [1, 2, 3, 4, 7, 13, 53])
def test_as_close_as_unfused(n):
    rng = np.random.default_rng(n)
    e = {"stated": 0.0, "unfused": 0.0}
    for _ in range(300):
        r = (-1 / (2 + 10.0 ** rng.uniform(-4, 1) + rng.uniform(0, 0.1, n))).astype(f)
        d = rng.standard_normal(n).astype(f)
        exact = 0.0
        for k in range(n):
            exact = float(r[k]) * (float(d[k]) - exact)
        e["stated"] += abs(float(_map(r, d, _fused(n))) - exact)
        e["unfused"] += abs(float(_map(r, d, [False] * n)) - exact)
    assert e["stated"] <= 1.05 * e["unfused"] + 1e-30
