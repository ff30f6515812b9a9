"""The integer conversions and comparisons of the FP64-accumulated step (csrc/f64bits.h) against the
host's IEEE conversions, bit for bit: ties, carries into the exponent, the ends of the accepted range
and random values."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include "f64bits.h"
using namespace cosmica::f64bits;
extern "C" {
void t_widen(const uint32_t *u, uint64_t *o, int n) { for (int i = 0; i < n; ++i) o[i] = widen(u[i]); }
void t_narrow(const uint64_t *u, uint32_t *o, int n) { for (int i = 0; i < n; ++i) o[i] = narrow(u[i]); }
void t_pi_minus(const uint64_t *u, float *o, int n) { for (int i = 0; i < n; ++i) o[i] = pi_minus(pi_minus_units(u[i])); }
void t_count(const uint32_t *u, uint64_t *o, int n) { for (int i = 0; i < n; ++i) o[i] = from_u32(u[i]); }
void t_cmp(const uint64_t *a, const uint64_t *b, uint8_t *l, uint8_t *oc, uint8_t *oh, uint8_t *fin, int n)
{ for (int i = 0; i < n; ++i) { l[i] = less(a[i], b[i]); oc[i] = outside_closed(a[i], b[i]);
    oh[i] = outside_half_open(a[i], b[i]); fin[i] = is_finite(a[i]); } }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("f64bits")
    (d / "t.cpp").write_text(SRC)
    subprocess.run(["g++", "-O1", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2502_06319_gb300", "csrc"),
                    str(d / "t.cpp"), "-o", str(d / "t.so")], check=True)
    return C.CDLL(str(d / "t.so"))


def p(a):
    return a.ctypes.data_as(C.c_void_p)


def test_widen(lib):
    rng = np.random.default_rng(1)
    u = np.concatenate([rng.integers(0, 2 ** 32, 200000, dtype=np.uint64).astype(np.uint32),
                        np.array([0, 0x80000000, 1, 0x007FFFFF, 0x00800000, 0x3F800000, 0x7F7FFFFF, 0x7F800000,
                                  0x7FC00000, 0xFF7FFFFF, 0xFF800000, 0x80800000], dtype=np.uint32)])
    o = np.empty(len(u), np.uint64)
    lib.t_widen(p(u), p(o), len(u))
    f = u.view(np.float32).copy()
    f[np.abs(f) < np.float32(2.0 ** -126)] *= np.float32(0.0)          # subnormals count as zero
    nan = np.isnan(f)
    assert np.array_equal(np.isnan(o.view(np.float64)), nan)
    assert np.array_equal(o[~nan], f[~nan].astype(np.float64).view(np.uint64))


def test_narrow(lib):
    rng = np.random.default_rng(2)
    x = np.exp(rng.uniform(-80, 80, 200000)) * np.where(rng.random(200000) < 0.5, -1, 1)
    f = np.abs(rng.standard_normal(50000)).astype(np.float32).view(np.uint32).astype(np.uint64)
    # halfway between two FP32 neighbours, and one unit to each side of it; carries into the exponent
    half = (np.uint32(0x38000000) + (f >> np.uint64(3)) << np.uint64(32)) + ((f & np.uint64(7)) << np.uint64(29)) + np.uint64(1 << 28)
    edge = np.array([2.0 ** -126, 2.0 ** -127, -2.0 ** -140, 2.0 ** -125, np.nextafter(2.0 ** -125, 0), 2.0 ** 127, np.nextafter(2.0 ** 127, 0), 0.0, -0.0, 1e-300,
                     1e300, np.inf, -np.inf, np.nan, np.nextafter(2.0, 0), np.nextafter(1.0, 0), -np.nextafter(4.0, 0)])
    u = np.concatenate([x.view(np.uint64), half, half + np.uint64(1), half - np.uint64(1), edge.view(np.uint64)])
    o = np.empty(len(u), np.uint32)
    lib.t_narrow(p(u), p(o), len(u))
    v = u.view(np.float64)
    with np.errstate(all="ignore"):
        f = v.astype(np.float32)
        f[np.abs(v) < 2.0 ** -126] *= np.float32(0.0)
        want = np.abs(v) < 2.0 ** 127
        assert np.array_equal(o[want], f[want].view(np.uint32))


def test_pi_minus(lib):
    rng = np.random.default_rng(3)
    th = np.concatenate([rng.uniform(np.pi / 2, np.pi, 200000), np.pi - np.exp(rng.uniform(-14, 0.4, 200000)),
                         np.array([np.pi / 2, np.pi, np.nextafter(np.pi, 0), 2.0, np.nextafter(2.0, 0), np.pi - 2.0 ** -20,
                                   np.pi - 2.0 ** -21])])
    o = np.empty(len(th), np.float32)
    lib.t_pi_minus(p(th.view(np.uint64)), p(o), len(th))
    assert np.array_equal(o, (np.pi - th).astype(np.float32))


def test_count(lib):
    rng = np.random.default_rng(5)
    u = np.concatenate([rng.integers(0, 2 ** 32, 50000, dtype=np.uint64), np.arange(40, dtype=np.uint64),
                        np.uint64(1) << np.arange(32, dtype=np.uint64), np.array([2 ** 32 - 1], dtype=np.uint64)]).astype(np.uint32)
    o = np.empty(len(u), np.uint64)
    lib.t_count(p(u), p(o), len(u))
    assert np.array_equal(o.view(np.float64), u.astype(np.float64))


def test_comparisons(lib):
    rng = np.random.default_rng(4)
    a = np.concatenate([rng.uniform(-10, 130, 100000), np.array([0.0, np.pi, 2 * np.pi, 122.0, 0.1, -1e-300, np.inf, -np.inf])])
    for b0 in (0.1, np.pi, 2 * np.pi, 122.0):
        b = np.full(len(a), b0)
        l, oc, oh, fin = (np.empty(len(a), np.uint8) for _ in range(4))
        lib.t_cmp(p(a.view(np.uint64)), p(b.view(np.uint64)), p(l), p(oc), p(oh), p(fin), len(a))
        assert np.array_equal(l.astype(bool), a < b)
        assert np.array_equal(oc.astype(bool), (a < 0) | (a > b))
        assert np.array_equal(oh.astype(bool), (a < 0) | (a >= b))
        assert np.array_equal(fin.astype(bool), np.isfinite(a))
    nan, one = np.array([np.nan, -np.nan]), np.ones(2)
    l, oc, oh, fin = (np.empty(2, np.uint8) for _ in range(4))
    lib.t_cmp(p(nan.view(np.uint64)), p(one.view(np.uint64)), p(l), p(oc), p(oh), p(fin), 2)
    assert not fin.any()
