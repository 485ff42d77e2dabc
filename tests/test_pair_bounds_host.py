"""The error bounds that the tensor-core pair scores state for their 16-bit parts, against an emulation
of the rounding in NumPy: x as hi + lo, the squares, the target's products, and the product left out."""
import os
import re

import numpy as np
import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2410_01752_gb300", "csrc", "pair_tc.cu")
U = 2.0 ** -24


def _stated(name):
    m = re.search(r"constexpr int [^;]*\b" + name + r" = (\d+)[,;]", open(SRC).read())
    assert m, name + " is not stated"
    return int(m.group(1)) * U


def _parts(x):
    """FP32 values in [-2^15, 2^15] as two FP16 parts, in FP64."""
    hi = x.astype(np.float16)
    lo = (x - hi.astype(np.float32)).astype(np.float16)
    return hi.astype(np.float64), lo.astype(np.float64)


@pytest.fixture(scope="module")
def rows():
    r = np.random.default_rng(0)
    x, g = (np.concatenate([r.uniform(1, 2, size=400000), 1 + r.integers(0, 2 ** 12, size=400000) * 2.0 ** -12 +
                            2.0 ** -12 * r.uniform(size=400000)]) * 2.0 ** 14 for _ in range(2))
    t = r.uniform(0.5, 1, size=x.size)
    r.shuffle(g)
    x32, g32, t32 = (v.astype(np.float32) for v in (x, g, t))
    return x, g, t, x32, g32, t32


def _relative(got, exact):
    return float(np.max(np.abs(got - exact) / np.abs(exact)))


def test_rows(rows):
    x, _, t, x32, _, t32 = rows
    hi, lo = _parts(x32)
    err = _relative(hi + lo, x)
    assert 2.0 * U < err <= _stated("kErrRow")
    sq = x32 * x32 * np.float32(2.0 ** -15)
    assert _relative(sum(_parts(sq)), x * x * 2.0 ** -15) <= _stated("kErrSquare")
    xr = (hi + lo).astype(np.float32) * t32
    assert _relative(sum(_parts(xr)), x * t) <= _stated("kErrTarget")


def test_products(rows):
    x, g, _, x32, g32, _ = rows
    xh, xl = _parts(x32)
    gh, gl = _parts(g32)
    assert float(np.max(np.abs(xl * gl) / (x * g))) <= _stated("kErrLoLo")
    kept = xh * gh + xh * gl + xl * gh
    assert _relative(kept, x * g) <= 2 * _stated("kErrRow") + _stated("kErrLoLo")
