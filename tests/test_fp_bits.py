"""The conversions between FP64 and FP32 by integer operations (csrc/fp_bits.cuh), compiled for the host,
against numpy's conversions, and the two FP32 screens of the FP64 forms with operands truncated by them:
a stencil that the fast form's test keeps is one that TENO5 keeps, and the screened maximum of the split
speeds is the exact one (the same stencils and blocks as with rounded operands).
"""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from oracle import oracle as O
from paper_1905_00182_gb300 import build as B
from tests import test_teno_shortcut as TS
from tests import test_wavespeed_screen as WS

HERE = os.path.dirname(os.path.abspath(__file__))
F = np.float32


@pytest.fixture(scope="module")
def bits(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no host compiler")
    out = str(tmp_path_factory.mktemp("bits") / "libfpbits.so")
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-I", B.CSRC,
                        os.path.join(HERE, "fp_bits_host.cpp"), "-o", out],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lib = ctypes.CDLL(out)

    def function(name, to):
        f = getattr(lib, name)
        f.argtypes = [ctypes.c_void_p, ctypes.c_void_p, ctypes.c_longlong]
        f.restype = None

        def call(x):
            x = np.ascontiguousarray(x, dtype=np.float32 if to is np.float64 else np.float64)
            y = np.empty(x.shape, dtype=to)
            f(x.ctypes.data, y.ctypes.data, x.size)
            return y

        return call

    return {"widen": function("widen_all", np.float64), "narrow": function("narrow_all", F),
            "low": function("low_precision_all", F)}


def _same(a, b):
    """equal bits, any NaN for a NaN"""
    u = np.uint64 if a.dtype == np.float64 else np.uint32
    return np.array_equal(np.isnan(a), np.isnan(b)) and np.array_equal(
        a.view(u)[~np.isnan(a)], b.view(u)[~np.isnan(b)])


def _floats():
    """FP32 numbers of every size and both signs: edges of the exponents, subnormals, a stride"""
    edge = (np.arange(256, dtype=np.uint32) << 23)[:, None] + np.arange(-70, 70)[None].astype(np.uint32)
    u = np.concatenate([edge.ravel() & 0x7FFFFFFF, np.arange(1 << 16, dtype=np.uint32),
                        np.uint32(1) << np.arange(31, dtype=np.uint32),
                        np.arange(0, 1 << 31, 1021, dtype=np.uint32)])
    return np.concatenate([u, u | 0x80000000]).astype(np.uint32).view(F)


def test_widen_is_the_conversion(bits):
    x = _floats()
    with np.errstate(invalid="ignore"):
        assert _same(bits["widen"](x), x.astype(np.float64))


def test_narrow_rounds_to_nearest_even(bits):
    rng = np.random.default_rng(1)
    f = _floats()
    f = f[np.isfinite(f)]
    with np.errstate(over="ignore", invalid="ignore", under="ignore"):
        up = np.nextafter(f, F(np.inf)).astype(np.float64)
        up[np.isinf(up)] = 2.0 ** 128
        tie = 0.5 * (f.astype(np.float64) + up)         # exact in FP64
        u = rng.integers(0, 1 << 64, 1 << 20, dtype=np.uint64)
        mid = (rng.integers(0x360, 0x490, 1 << 20).astype(np.uint64) << np.uint64(52)
               | u & np.uint64(0x800FFFFFFFFFFFFF))     # exponents around FP32's range
        x = np.concatenate([f.astype(np.float64), tie, np.nextafter(tie, np.inf),
                            np.nextafter(tie, -np.inf), u.view(np.float64), mid.view(np.float64),
                            [0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, -5e-324]])
        want, t = x.astype(F), tie.astype(F)
    assert _same(bits["narrow"](x), want)
    # the inputs meet every kind of result, and ties that round down and up
    assert np.isinf(want).any() and (want == 0).any() and (np.abs(want[want != 0]) < 2.0 ** -126).any()
    assert (t == f).sum() > 1000 and (t != f).sum() > 1000


def test_low_precision_truncates(bits):
    f = _floats()
    f = f[np.isfinite(f)]
    rng = np.random.default_rng(2)
    x = f.astype(np.float64) * (1.0 + rng.uniform(-2.0 ** -25, 2.0 ** -22, f.size))
    x = np.concatenate([f.astype(np.float64), x, [0.0, -0.0, 1e39, -1e300, np.inf, -np.inf, np.nan]])
    got = bits["low"](x)
    # truncated: the FP64 mantissa cut to FP32's 23 bits
    cut = (x.view(np.uint64) & np.uint64(0xFFFFFFFFE0000000)).view(np.float64)
    normal = (np.abs(cut) >= 2.0 ** -126) & (np.abs(cut) < 2.0 ** 128)
    assert np.array_equal(got[normal].astype(np.float64), cut[normal])
    assert (got[np.abs(x) < 2.0 ** -126] == 0).all()
    assert np.isnan(got[~(np.abs(x) < 2.0 ** 128)]).all()


def test_stencils_kept_with_truncated_differences(bits):
    rng = np.random.default_rng(7)
    V = np.array([np.asarray(v, dtype=np.float64) for v in TS._stencils(rng)])
    D = bits["low"](V[:, 1:] - V[:, :-1])
    kept = 0
    for v, d in zip(V, D):
        t = [d[1] - d[0], d[2] - d[1], d[3] - d[2]]
        u = [F(3) * d[1] - d[0], d[1] + d[2], d[3] - F(3) * d[2]]
        b = [F(13.0 / 3.0) * t[k] * t[k] + u[k] * u[k] for k in range(3)]
        if not abs(b[0] - b[2]) <= F(4) * min(b) + F(1.6e-29):
            continue
        kept += 1
        assert abs(O.teno5(v) - TS._linear(v)) <= 1e-14 * (np.max(np.abs(v)) + 1e-300), v
    assert 5000 < kept < len(V) - 2000


def test_screened_maximum_with_truncated_speeds(bits):
    rng = np.random.default_rng(11)
    for k, (ua, c2) in enumerate(WS._blocks(rng)):
        for scale in (1.0, 1e-13, 1e-19) if k % 8 == 0 else (1.0,):  # speeds of that size
            u, c = ua * scale, c2 * scale ** 2
            v32 = bits["low"](u) + np.sqrt(bits["low"](c))
            m32 = np.max(v32)
            far = F(0) if m32 < F(1e-12) else m32 * (F(1) - F(2e-6))
            exact = u + np.sqrt(c)
            assert np.max(np.where(~(v32 < far), exact, 0.0)) == np.max(exact)
