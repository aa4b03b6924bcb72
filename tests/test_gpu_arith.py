"""The library's own arithmetic against CUDA's, on the device and with the
library's compiler flags: the widening of FP32 values in the dot products for
all 2^32 arguments (bits equal; a NaN gives a NaN)."""
import ctypes
import os
import subprocess

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
