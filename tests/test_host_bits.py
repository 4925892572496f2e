"""The kernels' bit arithmetic (csrc/bits.cuh, compiled for the host) against exact integers and the
hardware's division and conversions."""
import ctypes
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    so = str(tmp_path_factory.mktemp("bits") / "host_bits.so")
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_1811_09821_gb300", "csrc"), os.path.join(ROOT, "tests", "host_bits.cpp"), "-o", so],
                   check=True)
    return ctypes.CDLL(so)


def call(fn, n, *arrays):
    fn(ctypes.c_long(n), *[a if isinstance(a, ctypes.c_int) else a.ctypes.data_as(ctypes.c_void_p) for a in arrays])


def test_reciprocal_is_the_division(lib):
    """Bit for bit 1.0 / d: random mantissas at every exponent, those next to 1 and 2 (the hard cases of a
    reciprocal's rounding), the ends of the range at which the kernel divides, subnormals, zeros, negative
    values, infinities and NaN."""
    rng = np.random.default_rng(0)
    exps = np.arange(2048, dtype=np.uint64)
    man = rng.integers(0, 1 << 52, (2048, 400), dtype=np.uint64)
    near = np.concatenate([np.arange(64), (1 << 52) - 1 - np.arange(64)]).astype(np.uint64)
    man = np.concatenate([man, np.broadcast_to(near, (2048, len(near)))], 1)
    b = ((exps[:, None] << np.uint64(52)) | man).ravel()
    b = np.concatenate([b, b | np.uint64(1 << 63)])
    d = b.view(np.float64)
    out = np.empty_like(d)
    call(lib.host_rcp, len(d), np.ascontiguousarray(d), out)
    with np.errstate(all="ignore"):
        want = 1.0 / d
    nan = np.isnan(want)
    assert np.array_equal(np.isnan(out), nan)
    assert np.array_equal(out.view(np.uint64)[~nan], want.view(np.uint64)[~nan])


@pytest.mark.parametrize("ex", [-1070, -1021, -30, 0, 1, 400, 1024])
def test_fixed_point_of_a_modulus(lib, ex):
    """floor(|v| 2^(56 - ex)) for |v| < 2^ex, both signs, down to subnormals and zero, as exact integers."""
    rng = np.random.default_rng(ex + 2000)
    top = min(ex + 1022, 2046)     # biased exponent of values just below 2^ex
    be = rng.integers(max(0, top - 120), max(1, top + 1), 500)
    bits = (be.astype(np.uint64) << np.uint64(52)) | rng.integers(0, 1 << 52, 500, dtype=np.uint64)
    if ex < -1021:                 # subnormal scale: values below 2^ex
        bits = rng.integers(0, 1 << (ex + 1074), 500, dtype=np.uint64)
    bits[:3] = 0, 1 << 63, 1
    if ex <= -1073:
        bits[2] = 0
    bits[::7] |= np.uint64(1 << 63)
    out = np.empty_like(bits)
    call(lib.host_fixed56, len(bits), bits, ctypes.c_int(ex), out)
    for b, o in zip(bits, out):
        v = abs(Fraction(float(np.uint64(b).view(np.float64))))
        assert v < Fraction(2) ** ex
        assert int(o) == int(v * Fraction(2) ** (56 - ex))


def test_level_sums_round_once(lib):
    """H 2^28 + L times 2^(ex - 70), |H| < 2^52 and |L| < 2^46, rounded to FP64 once: the nearest double of the
    exact value (Python's conversion of a fraction), ties and results below the normal range among them."""
    rng = np.random.default_rng(1)
    n = 6000
    mag = rng.integers(0, 52, n)
    H = (rng.integers(0, 1 << 52, n) >> mag) * rng.choice([-1, 1], n)
    L = (rng.integers(0, 1 << 46, n) >> rng.integers(0, 46, n)) * rng.choice([-1, 1], n)
    ex = rng.choice([0, 3, -40, -900, -1018, -1040, -1090, 1000], n).astype(np.int32)
    # ties: the 53 bits end in a half
    k = n // 4
    odd = rng.integers(1 << 52, 1 << 53, k)
    X = [int(o) * (1 << 20) + (1 << 19) + int(d) for o, d in zip(odd, rng.integers(-1, 2, k))]
    H[:k] = [x >> 28 for x in X]
    L[:k] = [x & ((1 << 28) - 1) for x in X]
    H[-5:], L[-5:] = [0, 0, 0, 1, -1], [0, 1, -1, -(1 << 28), 1 << 28]
    assert np.all(np.abs(H) < 1 << 52)
    out = np.empty(n, np.uint64)
    call(lib.host_levels, n, H.astype(np.int64), L.astype(np.int64), ex, out)
    got = out.view(np.float64)
    for i in range(n):
        x = Fraction(int(H[i]) * (1 << 28) + int(L[i])) * Fraction(2) ** (int(ex[i]) - 70)
        want = float(x)
        # below the normal range the 53 bits are rounded first (twice in all): one unit of the smallest double
        assert got[i] == want or (abs(want) < 2.0 ** -1022 and abs(got[i] - want) <= 2.0 ** -1074), (i, H[i], L[i], ex[i])


def test_split_pair_is_the_conversion(lib):
    """hi = fl32(v) and lo = fl32(v - hi) bit for bit, over every exponent an FP32 has and beyond, both signs,
    ties of either rounding, zeros, infinities and NaN."""
    rng = np.random.default_rng(2)
    e = np.repeat(np.arange(1023 - 160, 1023 + 135, dtype=np.uint64), 300)
    man = rng.integers(0, 1 << 52, len(e), dtype=np.uint64)
    man[::5] &= ~np.uint64((1 << 28) - 1)            # half a unit of hi
    man[1::5] = (man[1::5] & ~np.uint64((1 << 29) - 1)) | rng.integers(0, 1 << 6, len(man[1::5]), dtype=np.uint64)
    b = (e << np.uint64(52)) | man
    b[::2] |= np.uint64(1 << 63)
    special = np.array([0.0, -0.0, np.inf, -np.inf, 1e-310, 1.7e308]).view(np.uint64)
    b = np.concatenate([b, special])
    hi, lo = np.empty(len(b), np.float32), np.empty(len(b), np.float32)
    call(lib.host_split, len(b), b, hi, lo)
    v = b.view(np.float64)
    with np.errstate(all="ignore"):
        wh = v.astype(np.float32)
        wl = (v - wh.astype(np.float64)).astype(np.float32)
    np.testing.assert_array_equal(hi, wh)
    np.testing.assert_array_equal(lo, wl)
    nan = np.array([np.nan]).view(np.uint64)
    call(lib.host_split, 1, nan, hi, lo)
    assert np.isnan(hi[0]) and np.isnan(lo[0])
