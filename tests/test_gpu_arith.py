"""The library's own arithmetic against CUDA's, on the device and with the
library's compiler flags: the widening of FP32 values in the dot products for
all 2^32 arguments (bits equal; a NaN gives a NaN), and the corrected quotient
of the allocation-free solves.  The quotient can differ from the division, by one
ulp, only where t / d is within 2^-51 ulp of the middle between two doubles:
for random mantissas an event of probability 2^-50 a pair, so none of 2^23 differs."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def shim(tmp_path_factory):
    from paper_1312_1553_gb300 import _build

    out = tmp_path_factory.mktemp("shim") / "libarith.so"
    subprocess.run([_build._nvcc(), *_build.NVFLAGS, "-shared", os.path.join(HERE, "arith_shim.cu"), "-o", str(out)],
                   check=True)
    return ctypes.CDLL(str(out))


def test_wide_is_the_conversion(shim):
    bad = ctypes.c_ulonglong(1)
    assert shim.shim_wide(ctypes.byref(bad)) == 0
    assert bad.value == 0


def doubles(sign, exponent, mantissa):
    return (sign.astype(np.uint64) << 63 | (exponent + 1023).astype(np.uint64) << 52 | mantissa.astype(np.uint64)).view(
        np.float64)


def quotients(shim, t, d):
    q, div = np.empty_like(t), np.empty_like(t)
    assert shim.shim_quotient(len(t), *(ctypes.c_void_p(a.ctypes.data) for a in (t, d, q, div))) == 0
    return q, div


def test_quotient_random(shim):
    rng = np.random.default_rng(5)
    n = 1 << 23
    eq, ed = rng.integers(-498, 499, n), rng.integers(-332, 333, n)
    t = doubles(rng.integers(0, 2, n), np.clip(eq + ed, -1022, 1023), rng.integers(0, 1 << 52, n))
    d = doubles(rng.integers(0, 2, n), ed, rng.integers(0, 1 << 52, n))
    q, div = quotients(shim, t, d)
    np.testing.assert_array_equal(q.view(np.int64), div.view(np.int64))


def test_quotient_at_the_edges(shim):
    """Exponents on both sides of the two windows, mantissas at both ends of their range."""
    edge = np.concatenate([np.arange(4), (1 << 52) - 1 - np.arange(4), [1 << 51, (1 << 51) - 1]])
    ex = np.array([-1022, -1021, -970, -500, -499, -498, -497, -333, -332, -331, -1, 0, 1, 331, 332, 333, 497, 498, 499, 500,
                   970, 1022, 1023])
    et, mt, ed, md, sg = (a.ravel() for a in np.meshgrid(ex, edge, ex, edge, [0, 1], indexing="ij"))
    t, d = doubles(sg, et, mt), doubles(1 - sg, ed, md)
    q, div = quotients(shim, t, d)
    assert np.all(np.isinf(div) == np.isinf(q))
    assert np.abs(q.view(np.int64) - div.view(np.int64)).max() <= 1


def test_quotient_of_special_values(shim):
    v = np.array([0.0, -0.0, 5e-324, -5e-324, 2.2e-308, 2.3e-308, 1.0, -1.5, 1e300, -1e308, np.inf, -np.inf, np.nan])
    t, d = (np.ascontiguousarray(a.ravel()) for a in np.meshgrid(v, v))
    q, div = quotients(shim, t, d)
    np.testing.assert_array_equal(np.isnan(q), np.isnan(div))
    ok = ~np.isnan(div)
    np.testing.assert_array_equal(q[ok].view(np.int64), div[ok].view(np.int64))
