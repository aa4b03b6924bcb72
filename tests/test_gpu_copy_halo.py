"""The copying warps of the step form (copy_halo), alone on one CTA: all values
arrive whatever the length of the list; after a wait has run out the rest is
zeros without a further wait (nle.h: a solve that timed out finishes without
further waiting), however many values are missing."""
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

    out = tmp_path_factory.mktemp("shim") / "libcopyhalo.so"
    subprocess.run([_build._nvcc(), *_build.NVFLAGS, "-shared", os.path.join(HERE, "copy_halo_shim.cu"), "-o", str(out)],
                   check=True)
    return ctypes.CDLL(str(out))


def copy(shim, dtype, nh, missing, spin_ns):
    rng = np.random.default_rng(nh)
    x = rng.standard_normal(5000).astype(dtype)
    if missing:  # the not-yet-computed marker in every value
        x = (np.full(5000, 0xFFC0BAD1, np.uint32) if dtype == np.float32
             else np.full(5000, 0xFFF8BAD1BAD1BAD1, np.uint64)).view(dtype)
    hpos = rng.choice(5000, nh, replace=False).astype(np.int32)
    out, arrived, cycles, err = np.zeros(nh, dtype), np.zeros(4, np.int32), np.zeros(4, np.int64), np.zeros(1, np.int32)
    f = shim.shim_copy_f32 if dtype == np.float32 else shim.shim_copy_f64
    rc = f(ctypes.c_void_p(hpos.ctypes.data), nh, ctypes.c_void_p(x.ctypes.data), len(x),
           ctypes.c_longlong(spin_ns), *(ctypes.c_void_p(a.ctypes.data) for a in (out, arrived, cycles, err)))
    assert rc == 0 and np.all(arrived == nh)
    return x[hpos], out, int(cycles.max()), int(err[0])


@pytest.mark.parametrize("dtype,nh", [(t, n) for t in (np.float32, np.float64) for n in (1, 31, 33, 128, 129, 1000, 2047)])
def test_all_values_arrive(shim, dtype, nh):
    want, out, _, err = copy(shim, dtype, nh, False, 2_000_000_000)
    assert err == 0
    np.testing.assert_array_equal(out, want)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_no_wait_after_a_wait_ran_out(shim, dtype):
    """One chunk a warp (128 values) polls until the limit; 2,048 values are 16
    chunks a warp, of which only the first may wait."""
    _, out, one, err = copy(shim, dtype, 128, True, 1)
    assert err == 8 and not out.any()
    _, out, many, err = copy(shim, dtype, 2048, True, 1)
    assert err == 8 and not out.any()
    assert many < 3 * one
