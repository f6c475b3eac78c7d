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
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1403_7561_gb300", "csrc")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    tmp = tmp_path_factory.mktemp("arith")
    out = str(tmp / "libarith.so")
    (tmp / "cuda_runtime.h").write_text("")  # the harness defines what the headers take from it
    subprocess.run([gxx, "-O2", "-ffp-contract=off", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, "-I", str(tmp),
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


def test_split_rounds_to_46_bits(lib):
    rng = np.random.default_rng(3)
    a = rng.standard_normal(100000) * 2.0 ** rng.integers(-78, 120, 100000)
    edge = np.array([1.0, 2.0 - 2.0 ** -52, 1.0 + 2.0 ** -24 - 2.0 ** -52, 1.0 + 2.0 ** -47, 4.0 - 2.0 ** -51])
    a = np.concatenate([a, edge, -edge])
    bound = np.where(np.abs(a) >= 2.0 ** -80, 2.0 ** -47, 2.0 ** -23)  # the low word is dropped below 2^-80
    assert np.all(np.abs(call(lib.h_split, a, np.float64) - a) <= bound * np.abs(a))
    for v in (0.0, -0.0, np.inf, -np.inf):
        assert call(lib.h_split, np.array([v]), np.float64)[0] == v
    assert np.isnan(call(lib.h_split, np.array([np.nan]), np.float64)[0])


def test_grouped_sums_are_as_accurate_as_renormalized_steps(lib):
    # rows as the V stencil's: positive coefficients, vectors of both signs. The values are given 40
    # bits, so that they split exactly and the arithmetic is all that is measured
    rng = np.random.default_rng(5)
    n = 4000

    def bits40(v):
        m, e = np.frexp(v)
        return np.ldexp(np.round(np.ldexp(m, 40)), e - 40)

    c, x = bits40(rng.uniform(0.1, 1.0, (n, 27))), bits40(rng.standard_normal((n, 27)))
    g, s = np.empty(n), np.empty(n)
    lib.h_rows(n, *(v.ctypes.data_as(C.c_void_p) for v in (np.ascontiguousarray(c), np.ascontiguousarray(x), g, s)))
    exact = [sum(Fraction(a) * Fraction(b) for a, b in zip(c[i], x[i])) for i in range(n)]
    size = np.sqrt(np.mean(np.sum(c * np.abs(x), axis=1) ** 2))

    def rms(v):
        return np.sqrt(np.mean([float(Fraction(v[i]) - exact[i]) ** 2 for i in range(n)])) / size

    assert rms(g) <= 1.2 * rms(s), (rms(g), rms(s))


@pytest.mark.parametrize("groups", range(1, 9))
def test_fp32_gram_sums_at_most_32_rows(lib, groups):
    flush = lib.h_gram32_flush(groups)
    chunks = max(len(range(g, 8, groups)) for g in range(groups))  # of four rows, per tile and group
    assert 16 < 4 * chunks * flush <= 32


@pytest.mark.parametrize("devices,fails,want", [([0, 0, 1, 1, 0, 63, 63], 0, [1, 0, 1, 0, 0, 1, 0]),
                                                ([0, 0, 0, 1, 1], 1, [1, 1, 0, 1, 0]),
                                                ([-1, -1, 64, 64], 0, [1, 1, 1, 1])])
def test_function_attributes_are_set_on_every_device(lib, devices, fails, want):
    calls = (C.c_int * len(devices))()
    lib.h_once(len(devices), (C.c_int * len(devices))(*devices), fails, calls)
    assert list(calls) == want


@pytest.mark.parametrize("nx,ny,nz", [(1, 1, 1), (2, 2, 2), (64, 64, 32), (128, 128, 44), (500, 620, 7), (8192, 30, 9),
                                      (4, 4, 65535)])
def test_slabs_cover_every_plane_with_its_layers(lib, nx, ny, nz):
    slab = lib.h_slab_layers(nx, ny, nz)
    assert slab * 216 * nx * ny <= 64 << 20 or slab == min(2, nz)
    out = (C.c_int * (4 * (nz + 1)))()
    n = lib.h_slabs(nz, slab, nz + 1, out)
    rows = np.array(out).reshape(-1, 4)[:n]
    assert rows[0, 2] == 0 and rows[-1, 3] == nz + 1 and np.array_equal(rows[1:, 2], rows[:-1, 3])
    for e0, e1, p0, p1 in rows:
        assert 0 <= e0 < e1 <= nz and e1 - e0 <= slab and p0 < p1
        assert e0 <= max(p0 - 1, 0) and min(p1 - 1, nz - 1) < e1  # the layers below and above every plane
