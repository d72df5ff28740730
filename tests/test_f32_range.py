"""Which fp32 operands the tensor-core paths take (csrc/f32_range.h), on the CPU.

Whatever the rule accepts must come out of three bf16 planes and six plane
products with fp32's precision, on hardware that flushes subnormal planes and
products: the products are formed here in that way and compared with 64 bits.
What they cannot hold (infinities, NaN, 2^127, vectors or products that are too
small, sums that pass fp32's range) must be refused.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2607_20940_gb300", "csrc")

SOURCE = r"""
#include "f32_range.h"
extern "C" unsigned code(unsigned bits) { return msf::range_code(bits); }
extern "C" int holds(unsigned codes, int scale_exp) { return msf::range_holds(codes, scale_exp); }
extern "C" int gemm(unsigned a, unsigned b) { return msf::range_holds_gemm(a, b); }
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("f32_range")
    (d / "t.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-o", str(d / "t.so"), str(d / "t.cpp")],
                   check=True)
    return ctypes.CDLL(str(d / "t.so"))


def _code(rule, x, width=8):
    bits = np.abs(np.asarray(x, np.float32)).view(np.uint32).reshape(-1, width).max(1)
    return max(rule.code(int(b)) for b in np.unique(bits))


def _holds(rule, q, k, v, g=None, scale_exp=0):
    w = _code(rule, q) | _code(rule, k) << 8 | _code(rule, v) << 16
    return bool(rule.holds(w | (_code(rule, g) << 24 if g is not None else 0), scale_exp))


def _flush(x):
    return np.where(np.abs(x) < 2.0 ** -126, np.float32(0), x).astype(np.float32)


def _bf16(x):
    u = np.ascontiguousarray(x, np.float32).view(np.uint32)
    return ((u + np.uint32(0x7fff) + ((u >> np.uint32(16)) & np.uint32(1))) & np.uint32(0xffff0000)).view(np.float32)


def _planes(x):
    h = _bf16(x)
    m = _bf16(x - h)
    return [_flush(p) for p in (h, m, _bf16(x - h - m))]


def _product(x, y):
    """x y^T by six plane products, the small ones first, in fp32."""
    a, b = _planes(x), _planes(y)
    s = np.zeros((x.shape[0], y.shape[0]), np.float32)
    for i, j in ((0, 2), (1, 1), (0, 1), (2, 0), (1, 0), (0, 0)):
        for d in range(0, x.shape[1], 16):
            s += _flush(a[i][:, None, d:d + 16] * b[j][None, :, d:d + 16]).sum(2, dtype=np.float32)
    return s


def _operand(seed, rows, exp, spread=0):
    """Rows of 128 whose largest value has this exponent; with `spread`, neighbours differ by up to 2^spread."""
    r = np.random.default_rng(seed)
    x = r.uniform(1, 2, (rows, 128)) * r.choice([-1, 1], (rows, 128))
    if spread:
        x *= 2.0 ** -r.integers(0, spread, (rows, 128))
        x[:, ::8] = r.uniform(1, 2, (rows, 16))
    return (x * 2.0 ** exp).astype(np.float32)


@pytest.mark.parametrize("spread", [0, 40])
@pytest.mark.parametrize("uq,uk", [(0, 0), (58, 58), (116, 0), (-96, 96), (-96, -4), (-50, -50), (100, -96), (126, -96),
                                   (-10, 126)])
def test_accepted_scores_keep_fp32_precision(rule, uq, uk, spread):
    q, k, v = _operand(1, 24, uq, spread), _operand(2, 40, uk, spread), _operand(3, 40, 0)
    assert _holds(rule, q, k, v)
    s = _product(q, k)
    ref = q.astype(np.float64) @ k.astype(np.float64).T
    size = np.abs(q).astype(np.float64) @ np.abs(k).astype(np.float64).T
    # 48 fp32 additions of 16 products: 2^-24 of the running sum each
    assert np.isfinite(s).all() and (np.abs(s - ref) <= 48 * 2.0 ** -24 * size).all()


@pytest.mark.parametrize("uv,ug", [(0, 0), (-96, 26), (40, 40), (96, -96), (-30, -40)])
def test_accepted_gradients_keep_fp32_precision(rule, uv, ug):
    q, k = _operand(1, 16, 0), _operand(2, 24, 0)
    v, g = _operand(3, 24, uv), _operand(4, 16, ug)
    assert _holds(rule, q, k, v, g)
    dp = _product(g, v)
    ref = g.astype(np.float64) @ v.astype(np.float64).T
    size = np.abs(g).astype(np.float64) @ np.abs(v).astype(np.float64).T
    assert np.isfinite(dp).all() and (np.abs(dp - ref) <= 48 * 2.0 ** -24 * size).all()
    for p in (1.0, 2.0 ** -20):  # dS of probabilities near one, and of small ones
        ds = np.zeros((128, 16), np.float32)
        ds[:24] = (dp * np.float32(p)).T
        dk, ref = _product(ds.T, _operand(5, 8, 0)), ds.T.astype(np.float64) @ _operand(5, 8, 0).astype(np.float64).T
        size = np.abs(ds.T).astype(np.float64) @ np.abs(_operand(5, 8, 0)).astype(np.float64).T
        assert np.isfinite(dk).all() and (np.abs(dk - ref) <= 48 * 2.0 ** -24 * size).all()


def test_refused_forward(rule):
    one, zero = _operand(1, 16, 0), np.zeros((16, 128), np.float32)
    for bad in (np.inf, -np.inf, np.nan, 2.0 ** 127, np.finfo(np.float32).min):
        for where in range(3):
            x = [one.copy(), one.copy(), one.copy()]
            x[where][5, 17] = bad
            assert not _holds(rule, *x), (bad, where)
            x[where - 1] = zero  # also beside an operand of zeros
            assert not _holds(rule, *x), (bad, where)
    for where in range(3):  # a whole vector too small, whatever the rest is; single values and zeros may be
        for u in (-97, -118, -126, -140):
            x = [one.copy(), one.copy(), one.copy()]
            x[where][3, 8:16] = one[3, 8:16] * np.float32(2.0 ** u)
            assert not _holds(rule, *x), (u, where)
            x[where][3, 8] = 1
            assert _holds(rule, *x)
            x[where][3, 8:16] = 0
            assert _holds(rule, *x)
    assert _holds(rule, zero, zero, zero)
    s = np.float32
    assert not _holds(rule, one * s(2.0 ** 58), one * s(2.0 ** 59), one)   # scores past fp32
    assert not _holds(rule, one * s(2.0 ** -50), one * s(2.0 ** -51), one)  # scores too small
    assert not _holds(rule, one, one, one * s(2.0 ** 97))                  # sums of values past fp32
    assert _holds(rule, one * s(2.0 ** 100), one, one, scale_exp=16)       # scores past fp32 once scaled
    assert not _holds(rule, one * s(2.0 ** 100), one, one, scale_exp=17)
    assert _holds(rule, one * s(2.0 ** 100), one, one, scale_exp=-125)


def test_refused_gradient(rule):
    one, zero = _operand(1, 16, 0), np.zeros((16, 128), np.float32)

    def holds(q, k, v, g):
        return _holds(rule, *(one * np.float32(2.0 ** u) for u in (q, k, v, g)))

    assert holds(0, 0, 0, 0) and holds(0, 0, -35, -35) and holds(10, 10, 35, 35)
    assert not holds(0, 0, -35, -36)   # dP too small for dS's planes
    assert not holds(0, 0, 41, 40)     # dP too large
    assert not holds(0, 0, 0, 97) and not holds(0, 0, 0, -97)
    assert not holds(41, 0, 40, 0) and not holds(0, 41, 40, 0)      # dS q, dS k past the bound
    assert not holds(-20, 0, -35, -35) and not holds(0, -20, -35, -35)
    assert _holds(rule, one, one, one, zero) and _holds(rule, one, one, zero, one)


def test_gemm(rule):
    one = _operand(1, 4, 0)
    c = lambda u: _code(rule, one * np.float32(2.0 ** u), 4)  # noqa: E731
    assert rule.gemm(c(0), c(0)) and rule.gemm(c(52), c(53)) and rule.gemm(c(-50), c(-50)) and rule.gemm(0, c(120))
    assert not rule.gemm(c(53), c(53)) and not rule.gemm(c(-50), c(-51))
    assert not rule.gemm(c(0), c(-97)) and not rule.gemm(c(127), c(0)) and not rule.gemm(c(127), 0)
