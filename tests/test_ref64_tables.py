"""The FP64 filter's function tables as the build writes them, against extended precision."""
import os
import re

import numpy as np

from paper_2308_00763_gb300 import ref64_tables

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
LD = np.longdouble


def _numbers(row):
    return [float.fromhex(x.strip().rstrip("f") if "p" not in x else re.sub(r"f$", "", x.strip()))
            for x in row.strip("{}").split(",")]


def test_entries():
    hi, rest, lo, ex, ln, eln2 = [np.array([_numbers(e) for e in r]) for r in ref64_tables.rows()]
    assert [len(r) for r in (hi, rest, lo, ex, ln, eln2)] == [1024, 1024, 2048, 2048, 1024, 32]
    pi = LD("3.14159265358979323846264338327950288")
    a, b = pi * np.arange(1024) / 4096, pi * np.arange(2048) / 8388608
    # each value with its rest is good to about 2^-64 (the reference's own rounding)
    for k, f in ((0, np.cos), (1, np.sin)):
        assert np.abs(hi[:, k].astype(LD) + rest[:, k] - f(a)).max() < 2.0 ** -62
        assert np.abs(rest[:, k]).max() <= 2.0 ** -54
    assert np.abs(lo[:, 1] - np.sin(b)).max() <= 2.0 ** -64
    assert np.abs(lo[:, 0] + 2 * np.sin(b / 2) ** 2).max() <= 2.0 ** -75
    assert np.abs(ex[:, 0].astype(LD) + ex[:, 1] - np.exp2(np.arange(2048).astype(LD) / 2048)).max() < 2.0 ** -61
    c, low, high = ln.T
    j = np.arange(1024)
    want = -np.log(np.where(j >= ref64_tables.LN_UPPER, 2, 1) * c.astype(LD))
    assert np.abs(high.astype(LD) + low - want).max() < 2.0 ** -60
    assert np.array_equal(high * 2.0 ** 42, np.rint(high * 2.0 ** 42)) and np.abs(low).max() <= 2.0 ** -43
    # |z c - 1| <= 2^-11 over each interval of z (the last takes c = 1/2: z in [2 - 2^-10, 2))
    z0, z1 = 1 + j / 1024, 1 + (j + 1) / 1024
    assert max(np.abs(z0 * c - 1).max(), np.abs(z1 * c - 1).max()) <= 2.0 ** -11 * (1 + 2.0 ** -10)
    assert np.abs(eln2[:, 2].astype(LD) + eln2[:, 1] + np.log(LD(2)) * np.arange(32)).max() < 2.0 ** -58


def test_the_kernel_takes_the_same_line():
    with open(os.path.join(ROOT, "paper_2308_00763_gb300", "csrc", "pf_ref64.cuh")) as f:
        assert int(re.search(r"kLnUpper = (\d+);", f.read()).group(1)) == ref64_tables.LN_UPPER
