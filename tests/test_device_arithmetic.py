"""Device arithmetic that replaces FP64 instructions, compiled for the host (CPU).

The headers fpbits.cuh and dfloat.cuh are compiled from the library's own source with host
definitions of the few intrinsics they use (arith_harness.cpp) and compared with the plain
operations over all classes of values: zeros, subnormals, both ends of the normal range,
infinities and NaN.
"""
import ctypes as C
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1403_7561_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    out = str(tmp_path_factory.mktemp("arith") / "libarith.so")
    subprocess.run([gxx, "-O2", "-ffp-contract=off", "-std=c++17", "-shared", "-fPIC", "-I", CSRC,
                    os.path.join(ROOT, "tests", "arith_harness.cpp"), "-o", out], check=True, capture_output=True)
    return C.CDLL(out)


def call(f, a, dtype):
    out = np.empty(len(a), dtype=dtype)
    f(len(a), a.ctypes.data_as(C.c_void_p), out.ctypes.data_as(C.c_void_p))
    return out


def patterns():
    """Every exponent with both signs and a few mantissas, the special values, random patterns."""
    e = np.arange(2048, dtype=np.uint64) << np.uint64(52)
    m = np.array([0, 1, 1 << 28, 1 << 29, (1 << 52) - 1, 0x5555555555555], dtype=np.uint64)
    a = (e[:, None] | m[None, :]).ravel()
    rng = np.random.default_rng(7)
    a = np.concatenate([a, a | np.uint64(1 << 63), rng.integers(0, 1 << 64, 200000, dtype=np.uint64)])
    return a.view(np.float64)


@pytest.mark.parametrize("name,dtype,ref", [("h_times4", np.float64, lambda a: 4.0 * a),
                                            ("h_d2f", np.float32, lambda a: a.astype(np.float32))])
def test_bit_operations_equal_the_plain_ones(lib, name, dtype, ref):
    a = patterns()
    with np.errstate(all="ignore"):
        want = ref(a)
    got = call(getattr(lib, name), a, dtype)
    nan = np.isnan(want)
    assert np.array_equal(np.isnan(got), nan)
    u = np.uint64 if dtype == np.float64 else np.uint32
    assert np.array_equal(got[~nan].view(u), want[~nan].view(u))
