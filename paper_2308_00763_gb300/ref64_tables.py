"""The tables of the FP64 filter's elementary functions (``csrc/pf_ref64.cuh``) as a C++ initialiser.

Every entry is rounded once from 60 decimal digits, so the file is the same on every machine.
The build writes it next to the objects; compiled in as initialised data, the tables are there in
every CUDA context that loads the library, without an upload or any state in the process.
"""
from __future__ import annotations

import os
import struct
from decimal import ROUND_HALF_EVEN, Decimal, localcontext

PI = Decimal("3.14159265358979323846264338327950288419716939937510582097494459")
LN_UPPER = 424   # first logarithm interval whose centre is above sqrt 2 (kLnUpper)


def _sin_cos(a: Decimal):
    """Sine and cosine of 0 <= a < 1 by their power series."""
    s, c, term, k = Decimal(0), Decimal(0), Decimal(1), 0
    while abs(term) > Decimal("1e-58"):
        sign = -1 if k & 2 else 1
        if k & 1:
            s += sign * term
        else:
            c += sign * term
        k += 1
        term = term * a / k
    return s, c


def _f32(x) -> float:
    return struct.unpack("f", struct.pack("f", float(x)))[0]


def _pair(a: float, b: float) -> str:
    return "{%s, %s}" % (a.hex(), b.hex())


def _with_rest(v: Decimal):
    hi = float(v)
    return hi, v - Decimal(hi)


def _ln(c: float, v: Decimal) -> str:
    """{c, rest, multiple of 2^-42 nearest to v}"""
    unit = Decimal(2) ** 42
    hi = (v * unit).quantize(Decimal(1), rounding=ROUND_HALF_EVEN) / unit
    return "{%sf, %sf, %s}" % (c.hex(), _f32(v - hi).hex(), float(hi).hex())


def rows():
    """The members of Ref64Tables in order, each a list of entries."""
    with localcontext() as ctx:
        ctx.prec = 60
        return _rows()


def _rows():
    hi, hi_rest = [], []
    for i in range(1024):
        s, c = _sin_cos(PI * i / 4096)
        (c0, c1), (s0, s1) = _with_rest(c), _with_rest(s)
        hi.append(_pair(c0, s0))
        hi_rest.append("{%sf, %sf}" % (_f32(c1).hex(), _f32(s1).hex()))
    lo = []
    for i in range(2048):
        s, _ = _sin_cos(PI * i / 8388608)
        h, _ = _sin_cos(PI * i / 16777216)
        lo.append(_pair(float(-2 * h * h), float(s)))
    ln2 = Decimal(2).ln()
    ex = []
    for i in range(2048):
        v, rest = _with_rest((ln2 * i / 2048).exp())
        ex.append(_pair(v, float(rest)))
    ln = []
    for j in range(1024):
        # the last interval takes c = 1/2, so that ln u keeps its relative accuracy next to u = 1
        c = 0.5 if j == 1023 else _f32(1.0 / (1.0 + (j + 0.5) / 1024))
        ln.append(_ln(c, -(Decimal(c) * (2 if j >= LN_UPPER else 1)).ln()))
    eln2 = [_ln(0.0, -ln2 * i) for i in range(32)]
    return [hi, hi_rest, lo, ex, ln, eln2]


def write(path: str) -> str:
    text = ",\n".join("{%s}" % ",\n".join(r) for r in rows()) + "\n"
    tmp = path + ".tmp%d" % os.getpid()
    with open(tmp, "w") as f:
        f.write(text)
    os.replace(tmp, path)
    return path
