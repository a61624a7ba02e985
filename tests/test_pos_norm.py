"""The norm of a positional step as fixed-point shares (`qw_pos_norm.h`): the header
is compiled here with the host C++ compiler (no CUDA) and its sums, as the
grid's barrier words and a cluster's two sums hold them, are compared with
exact integers and fractions, for norms from 0 to 2^17 times the target, targets
from subnormal to the largest, and shares that no integer sum takes."""
import ctypes
import math
import os
import shutil
import subprocess
from decimal import Decimal, getcontext
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_2303_06890_gb300", "csrc")

SHIM = r"""
#include "qw_pos_norm.h"
extern "C" {
int unit_exp(double t) { return pos_unit_exp(t); }
uint64_t units(double v, int k, int *odd) { bool o; const uint64_t u = pos_units(v, k, o); *odd = o; return u; }
int deviation56(uint64_t t, uint64_t f, uint64_t c, int64_t *d) { *d = pos_deviation<56>(t, f); return pos_near(t, c); }
int deviation64(uint64_t t, uint64_t f, uint64_t c, int64_t *d) { *d = pos_deviation<64>(t, f); return pos_near(t, c); }
int factor(int64_t dev, float ih, float il, float *h, float *l) { return pos_factor_pair(dev, ih, il, *h, *l); }
void split(double v, float *h, float *l) { factor_split(v, *h, *l); }
double total56(uint64_t f, uint64_t c, double x, int k) { return pos_total<56>(f, c, x, k); }
double total64(uint64_t f, uint64_t c, double x, int k) { return pos_total<64>(f, c, x, k); }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    d = tmp_path_factory.mktemp("posnorm")
    (d / "shim.cpp").write_text(SHIM)
    so = str(d / "libnorm.so")
    subprocess.run([cxx, "-std=c++17", "-O1", "-shared", "-fPIC", "-I", CSRC, str(d / "shim.cpp"), "-o", so], check=True)
    lib = ctypes.CDLL(so)
    u64, i64, f64, i32 = ctypes.c_uint64, ctypes.c_int64, ctypes.c_double, ctypes.c_int
    lib.unit_exp.argtypes = [f64]
    lib.units.argtypes, lib.units.restype = [f64, i32, ctypes.POINTER(i32)], u64
    f32 = ctypes.c_float
    lib.split.argtypes = [f64, ctypes.POINTER(f32), ctypes.POINTER(f32)]
    lib.factor.argtypes = [i64, f32, f32, ctypes.POINTER(f32), ctypes.POINTER(f32)]
    for n in (56, 64):
        getattr(lib, f"deviation{n}").argtypes = [u64, u64, u64, ctypes.POINTER(i64)]
        f = getattr(lib, f"total{n}")
        f.argtypes, f.restype = [u64, u64, f64, i32], f64
    return lib


def _units(lib, v, k):
    odd = ctypes.c_int()
    u = lib.units(v, k, ctypes.byref(odd))
    return u, bool(odd.value)


def _sums(lib, shares, k, field):
    """The two words' sums of the blocks' shares, an FP64 sum of the odd ones, and
    the exact sum in units; a block is 16 warps of 32 lanes."""
    fine = coarse = count = exact = 0
    extra = 0.0
    for block in shares:
        f = c = 0
        odd = False
        for warp in block:
            w = 0
            for v in warp:
                u, o = _units(lib, v, k)
                odd |= o
                w += u
            f, c = (f + w) % 2**64, c + (w >> 42)
        if odd:
            extra += float(np.sum([np.sum(w) for w in block]))
            f, c = 0, 2**48
        else:
            exact += sum(_units(lib, v, k)[0] for w in block for v in w)
        if field == 56:  # the words of the barrier
            fine, coarse, count = (fine + (f << 8) + 1) % 2**64, (coarse + (c << 8) + 1) % 2**64, count + 1
            assert fine & 255 == coarse & 255 == count  # whatever the norm is
        else:
            fine, coarse = (fine + f) % 2**64, coarse + c
    return (fine >> 8, coarse >> 8, extra, exact) if field == 56 else (fine, coarse, extra, exact)


@pytest.mark.parametrize("target", [1.0, 0.3, 1.999, 2.0**-100, 1e-30, 1e-300, 5e-324, 3e-310, 1e30, 1.7e308])
def test_units_hold_the_target(lib, target):
    k = lib.unit_exp(target)
    u, odd = _units(lib, target, k)
    if target < 2.3e-308:  # the shares of a subnormal target are summed in FP64
        assert odd
    else:
        assert not odd and 2**61 <= u < 2**62 and u == Fraction(target) * Fraction(2) ** k
    assert _units(lib, 4.0 * target, k)[1] and _units(lib, 0.0, k) == (0, False)


@pytest.mark.parametrize("target", [0.0, -1.0, math.inf, math.nan])
def test_a_target_without_units_leaves_the_sum_to_fp64(lib, target):
    k = lib.unit_exp(target)
    for v in (5e-324, 1e-300, 1.0, math.inf, math.nan):
        assert _units(lib, v, k) == (0, True)
    assert _units(lib, 0.0, k) == (0, False)


@pytest.mark.parametrize("v", [1.0, 0.7, 2.0**-62, 2.0**-63, 1.5 * 2.0**-62, 1e-17, 1.9999, 3.9])
def test_units_round_to_nearest(lib, v):
    u, odd = _units(lib, v, 61)
    assert odd == (v >= 4.0) and abs(Fraction(u) - Fraction(v) * 2**61) <= Fraction(1, 2)


@pytest.mark.parametrize("field", [56, 64])
@pytest.mark.parametrize("ratio", [0.0, 1e-9, 0.5, 1.0 - 2.0**-30, 1.0, 1.0 + 2.0**-24, 2.0, 3.9, 4.0, 8.0, 64.0, 2.0**17])
@pytest.mark.parametrize("blocks", [1, 152, 255])
def test_sums_of_any_norm(lib, field, ratio, blocks):
    """`ratio` times the target in equal and in random shares: counts are whole, the
    norm is the exact sum's to an FP64 rounding or two, the deviation from the target
    is exact wherever it is reported, and it is wherever the norm is near."""
    blocks = min(blocks, 16) if field == 64 else blocks
    rng = np.random.default_rng(blocks)
    target = 0.37
    k = lib.unit_exp(target)
    t_units, _ = _units(lib, target, k)
    for equal in (True, False):
        v = np.ones((blocks, 2, 3)) if equal else rng.random((blocks, 2, 3))
        v *= ratio * target / v.sum()
        fine, coarse, extra, exact = _sums(lib, v, k, field)
        got = getattr(lib, f"total{field}")(fine, coarse, extra, k)
        want = Fraction(exact) / Fraction(2) ** k + Fraction(extra)
        assert abs(Fraction(got) - want) <= want * Fraction(3, 2**53)
        assert abs(got - ratio * target) <= 1e-14 * ratio * target + v.size * 2.0**-62 * target
        dev = ctypes.c_int64()
        if getattr(lib, f"deviation{field}")(t_units, fine, coarse, ctypes.byref(dev)):
            assert extra == 0.0 and dev.value == t_units - exact
        else:
            assert abs(ratio - 1.0) > 1e-4


def test_a_lane_beyond_the_integers_is_summed_in_fp64(lib):
    k = lib.unit_exp(1.0)
    v = np.full((4, 2, 3), 0.01)
    v[2, 1, 0] = 1e6
    fine, coarse, extra, _ = _sums(lib, v, k, 56)
    assert not lib.deviation56(_units(lib, 1.0, k)[0], fine, coarse, ctypes.byref(ctypes.c_int64()))
    assert lib.total56(fine, coarse, extra, k) == pytest.approx(v.sum(), rel=1e-15)
    v[2, 1, 0] = math.nan
    fine, coarse, extra, _ = _sums(lib, v, k, 56)
    assert math.isnan(lib.total56(fine, coarse, extra, k))


@pytest.mark.parametrize("target", [2**61, 2**61 + 12345678901, 3 * 2**60 + 7, 2**62 - 1])
def test_factor_as_a_float_pair(lib, target):
    """h + l is sqrt(target / sum) to 2^-48, h its rounding to FP32 or a neighbour, up to
    2^-14 from the target (in 60-digit decimal arithmetic)."""
    getcontext().prec = 60
    rng = np.random.default_rng(target % 1000)
    inv = 2.0**24 / target
    ih = np.float32(inv)
    il = np.float32(inv - float(ih))
    devs = [0, 1, -1, 2**24, 2**24 - 1, -2**24, 2**47 - 1, -2**47]
    devs += [int(s * 2.0**e) for e in rng.uniform(0, 47, 3000) for s in (1, -1)]
    h, l = ctypes.c_float(), ctypes.c_float()
    for dev in devs:
        assert lib.factor(dev, ih, il, ctypes.byref(h), ctypes.byref(l))
        want = (Decimal(target) / Decimal(target - dev)).sqrt()
        assert abs(Decimal(h.value) + Decimal(l.value) - want) <= Decimal(2) ** -48
        assert abs(l.value) <= 2.0**-23
    for dev in (2**47, -2**47 - 1, 2**54):
        assert not lib.factor(dev, ih, il, ctypes.byref(h), ctypes.byref(l))


def test_a_factor_keeps_48_bits(lib):
    """The float pair a factor is applied as: 2^-48 of it at any distance from 1."""
    h, l = ctypes.c_float(), ctypes.c_float()
    rng = np.random.default_rng(0)
    for v in [1.0, 1.0 + 2.0**-30, *(1.0 + s * 2.0**-e for e in rng.uniform(1, 50, 2000) for s in (1, -1)), 1e-3, 700.3]:
        lib.split(v, ctypes.byref(h), ctypes.byref(l))
        assert abs(Fraction(h.value) + Fraction(l.value) - Fraction(v)) <= Fraction(v) / 2**48
        assert h.value == np.float32(v)
