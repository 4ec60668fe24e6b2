"""The strict FP64 form's TENO5 without its weights' divisions, checked against the oracle's TENO5
on the CPU (arXiv:1905.00182, Sec. 2; the cut-off of TENO5).

The strict form looks TENO5's weights up where a sufficient test, taken in FP32 on the stencil's
FP64 first differences (truncated to FP32), proves that every stencil is kept, and where the
stencil is constant; everything else goes through the full evaluation.  The result must be the
oracle's to the bit, so what has to hold is: wherever one of the two rules applies, the oracle's
TENO5 equals the candidates combined with the looked-up weights, rounded in the oracle's order.
The rules are written out here in numpy and run on smooth, rough and tiny stencils, on stencils of
rounding noise around a constant (the oracle's indicators are then rounding themselves: without
the test's floor of (2e-13 c)^2 this fails), on exact constants and at the cut-off.
"""
import os
import sys

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)

from oracle import oracle as O  # noqa: E402

F = np.float32


def _trunc(x):
    """FP64 -> FP32 by truncation, 0 below and NaN above FP32's normal range"""
    if x == 0.0 or abs(x) < 2.0 ** -126:
        return F(0)
    if abs(x) >= 2.0 ** 127:
        return F(np.nan)
    m, e = np.frexp(x)
    return F(np.ldexp(np.trunc(np.ldexp(m, 24)), int(e) - 24))


def _mask(v, floor=True):
    """7 / 3 where a rule applies, None where the full evaluation decides"""
    d64 = [v[k + 1] - v[k] for k in range(4)]
    d = [_trunc(x) for x in d64]
    with np.errstate(over="ignore", invalid="ignore", under="ignore"):
        t = [d[1] - d[0], d[2] - d[1], d[3] - d[2]]
        u = [F(3) * d[1] - d[0], d[1] + d[2], d[3] - F(3) * d[2]]
        b = [F(13.0 / 3.0) * t[k] * t[k] + u[k] * u[k] for k in range(3)]
        m, c = min(b), _trunc(v[2])
        low = max(F(1e-35), F(4e-26) * c * c) if floor else F(0)
        if abs(b[0] - b[2]) <= F(4) * m and m >= low:
            return 7
    if all(x == 0.0 for x in d64):
        r = 3.0 * v[2] - 4.0 * v[2] + v[2]
        return 7 if r == 0.0 else 3 if abs(r) > 1e-18 else None
    return None


def _value(v, mask):
    a, b, c, d, e = v
    lin = [x if (mask >> k) & 1 else 0.0 for k, x in enumerate((0.1, 0.6, 0.3))]
    s = lin[0] + lin[1] + lin[2]
    w = [x / s for x in lin]
    q0 = (2.0 * a - 7.0 * b + 11.0 * c) / 6.0
    q1 = (-b + 5.0 * c + 2.0 * d) / 6.0
    q2 = (2.0 * c + 5.0 * d - e) / 6.0
    return w[0] * q0 + w[1] * q1 + w[2] * q2


def _stencils(rng, n=4000):
    x = np.arange(5, dtype=np.float64)
    for _ in range(n):
        off, scale = rng.normal() * 10.0 ** rng.uniform(-3, 2), 10.0 ** rng.uniform(-17, 0)
        c = rng.normal(size=4)
        yield off + scale * (c[0] * x + c[1] * x ** 2 + c[2] * x ** 3
                             + 10.0 ** rng.uniform(-6, 0) * rng.normal(size=5))
        yield rng.normal(size=5) * 10.0 ** rng.uniform(-40, 1)
        yield rng.normal() + 10.0 ** rng.uniform(-17, -10) * rng.normal(size=5)  # rounding noise
        s = np.zeros(5)
        s[rng.integers(1, 5):] = 10.0 ** rng.uniform(-16, 0)
        yield rng.normal() + s
        yield np.full(5, rng.normal() * 10.0 ** rng.uniform(-30, 3))
        # near the cut-off: linear middle, the outer indicators growing apart
        yield (off + scale * np.array([rng.uniform(-3, 3), 1.0, 2.0, 3.0, rng.uniform(0, 8)]))


def test_shortcut_gives_the_oracles_bits():
    rng = np.random.default_rng(5)
    used = {7: 0, 3: 0}
    for v in _stencils(rng):
        v = [float(x) for x in v]
        m = _mask(v)
        if m is None:
            continue
        used[m] += 1
        assert _value(v, m) == O.teno5(v), (v, m)
    assert used[7] > 1000 and used[3] > 100


def test_floor_is_needed():
    rng = np.random.default_rng(6)
    bad = 0
    for v in _stencils(rng, 2000):
        v = [float(x) for x in v]
        if _mask(v) is None and _mask(v, floor=False) == 7:
            bad += _value(v, 7) != O.teno5(v)
    assert bad > 0
