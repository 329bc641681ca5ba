"""The library's own bit-pattern functions (csrc/fempic_bits.cuh), compiled for
the host: conversions against the compiler's over the whole range, fallbacks
included; the refined reciprocal in ulps and the exit face against the choice by
FP64 quotients, each with the FP32 quotient they start from off by up to the two
ulps a device's approximate division is allowed."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2208_12795_gb300", "csrc")
HARNESS = r"""
#include <math.h>
#include <stdint.h>
#include <string.h>
static int off_ulps = 0;   // what the quotient is off by
static inline float off_div(float a, float b) {
  if (fabsf(b) > 0x1p126f) return isfinite(a) ? 0.0f : NAN;   // as the approximate division documents
  float q = a / b;
  if (q == 0.0f || !isfinite(q)) return q;
  for (int i = 0; i < (off_ulps < 0 ? -off_ulps : off_ulps); i++) q = nextafterf(q, off_ulps < 0 ? 0.0f : INFINITY);
  return q;
}
#define FEMPIC_HOST_FAST_DIV(a, b) off_div(a, b)
#include "fempic_bits.cuh"
using namespace fempic;
extern "C" {
void set_off(int u) { off_ulps = u; }
#define EACH(name, R, T, call) void name(int64_t n, const T* a, R* o) { for (int64_t i = 0; i < n; i++) o[i] = call(a[i]); }
EACH(t_f32_to_f64, double, float, f32_to_f64)
EACH(t_widen32, double, float, widen32)
EACH(t_f64_to_f32, float, double, f64_to_f32)
EACH(t_trunc32, float, double, trunc32)
EACH(t_recip_ge1, double, double, recip_ge1)
EACH(t_finite, uint8_t, double, finite_bits)
EACH(t_negative, uint8_t, double, negative_bits)
void t_split(int64_t n, const double* a, float* hi, float* lo) {
  for (int64_t i = 0; i < n; i++) { FF f = split_f64(a[i]); hi[i] = f.hi; lo[i] = f.lo; }
}
void t_exit(int64_t n, const double* la, const double* lb, const int32_t* entry, int32_t* k, double* s) {
  for (int64_t i = 0; i < n; i++) k[i] = exit_face64(la + 4 * i, lb + 4 * i, entry[i], s[i]);
}
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("bits")
    src, so = d / "bits.cpp", d / "libbits.so"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared", "-Wno-unknown-pragmas",
                    "-I", CSRC, str(src), "-o", str(so)], check=True)
    return C.CDLL(str(so))


def _call(lib, name, a, out_dtype):
    a = np.ascontiguousarray(a)
    o = np.empty(a.shape, out_dtype)
    getattr(lib, name)(C.c_int64(a.size), a.ctypes.data_as(C.c_void_p), o.ctypes.data_as(C.c_void_p))
    return o


def _doubles():
    rng = np.random.default_rng(3)
    f = np.abs(rng.standard_normal(5000)).astype(np.float32)
    up = np.nextafter(f, np.float32(np.inf)).astype(np.float64)
    mid = (f.astype(np.float64) + up) / 2
    wide = rng.random(40000) * 2.0 ** rng.uniform(-160, 140, 40000)
    edge = np.array([0.0, 2.0 ** -1074, 2.0 ** -150, 2.0 ** -149, 2.0 ** -127, 2.0 ** -126, 2.0 ** 127, 2.0 ** 128,
                     np.finfo(np.float32).max, np.finfo(np.float64).max, np.inf, np.nan, 1 - 2.0 ** -25, 1.0])
    with np.errstate(over="ignore"):
        edge = np.concatenate([edge, np.nextafter(edge, 0), np.nextafter(edge, np.inf)])
    v = np.concatenate([wide, mid, np.nextafter(mid, 0), np.nextafter(mid, 9.0), f.astype(np.float64), edge])
    return np.concatenate([v, -v])


def _floats():
    rng = np.random.default_rng(4)
    u = rng.integers(0, 2 ** 32, 60000, dtype=np.uint64).astype(np.uint32)
    edge = np.array([0, 1, 0x7fffff, 0x800000, 0x7f7fffff, 0x7f800000, 0x7fc00000], np.uint32)
    u = np.concatenate([u, edge, edge | np.uint32(0x80000000)])
    return u.view(np.float32)


@pytest.mark.parametrize("name", ["t_f32_to_f64", "t_widen32"])
def test_widening(lib, name):
    f = _floats()
    with np.errstate(invalid="ignore"):
        want = f.astype(np.float64)
    got = _call(lib, name, f, np.float64)
    nan = np.isnan(want)
    assert np.array_equal(np.isnan(got), nan)
    assert np.array_equal(got[~nan].view(np.uint64), want[~nan].view(np.uint64))


def test_rounding(lib):
    r = _doubles()
    with np.errstate(over="ignore", invalid="ignore"):
        want = r.astype(np.float32)
    got = _call(lib, "t_f64_to_f32", r, np.float32)
    nan = np.isnan(want)
    assert np.array_equal(np.isnan(got), nan)
    assert np.array_equal(got[~nan].view(np.uint32), want[~nan].view(np.uint32))


def test_truncation_and_split(lib):
    r = _doubles()
    f = _call(lib, "t_trunc32", r, np.float32)
    a = np.abs(r)
    small, big = a < 2.0 ** -126, ~(a < 2.0 ** 128)      # NaN counts as big
    mid = ~small & ~big
    assert (f[small] == 0).all() and np.isinf(f[big]).all()
    fd = f[mid].astype(np.float64)
    assert np.all(np.abs(fd) <= a[mid]) and np.all(a[mid] - np.abs(fd) <= a[mid] * 2.0 ** -23)
    assert np.array_equal(np.signbit(fd), np.signbit(r[mid]))
    hi, lo = np.empty(r.size, np.float32), np.empty(r.size, np.float32)
    lib.t_split(C.c_int64(r.size), r.ctypes.data_as(C.c_void_p), hi.ctypes.data_as(C.c_void_p),
                lo.ctypes.data_as(C.c_void_p))
    assert np.array_equal(hi[mid], f[mid]) and not hi[~mid].any() and not lo[~mid].any()
    # the low part keeps 24 of the remaining 29 bits where its scale is a normal float (exponents above -75)
    ok = mid & (a >= 2.0 ** -74)
    err = np.abs(r[ok] - (hi[ok].astype(np.float64) + lo[ok].astype(np.float64)))
    assert np.all(err <= a[ok] * 2.0 ** -47)


def test_signs_and_finiteness(lib):
    r = _doubles()
    assert np.array_equal(_call(lib, "t_finite", r, np.uint8).astype(bool), np.isfinite(r))
    fin = r[~np.isnan(r)]
    assert np.array_equal(_call(lib, "t_negative", fin, np.uint8).astype(bool), fin < 0)


@pytest.mark.parametrize("off", [-2, -1, 0, 1, 2])
def test_reciprocal(lib, off):
    """The seed is off by at most 2^-23 (truncation) + 2 ulp (2^-22), e below 2^-21.4, so the series' remainder
    e^3 is below 2^-64 of the result, 2^-11 of its ulp; the rest is the last multiply-add's half ulp."""
    if np.finfo(np.longdouble).nmant < 63:
        pytest.skip("needs a long double wider than a double")
    rng = np.random.default_rng(5)
    w = np.concatenate([1 + rng.random(40000) * 2.0 ** rng.uniform(-52, 10, 40000), 2.0 ** rng.uniform(0, 300, 40000),
                        2.0 ** np.arange(0, 140), np.nextafter(2.0 ** np.arange(1, 140), 0),
                        np.nextafter(2.0 ** np.arange(0, 140), np.inf)])
    lib.set_off(off)
    got = _call(lib, "t_recip_ge1", w, np.float64)
    lib.set_off(0)
    exact = np.longdouble(1) / w.astype(np.longdouble)
    ulp = np.spacing(exact.astype(np.float64))
    err = np.abs((got.astype(np.longdouble) - exact) / ulp)
    assert err.max() <= 0.5 + 2.0 ** -9, float(err.max())
    assert np.array_equal(_call(lib, "t_recip_ge1", np.array([np.inf, np.nan]), np.float64), [0.0, np.nan],
                          equal_nan=True)


def _pieces(kind, n=40000):
    """(la, lb): barycentrics of a piece's start and end."""
    rng = np.random.default_rng(6)
    la = rng.dirichlet(np.ones(4), n)
    d = rng.standard_normal((n, 4))
    lb = la + (d - d.mean(1, keepdims=True)) * 2.0 ** rng.uniform(-6, 3, (n, 1))
    if kind == "ties":        # two faces left at nearly the same fraction of the way
        s = rng.random(n) * 0.9 + 0.05
        off = np.where(rng.random(n) < 0.1, 0.0, rng.choice([-1, 1], n) * 2.0 ** rng.uniform(-54, -14, n))
        for k, f in ((1, s), (2, s * (1 + off))):
            lb[:, k] = la[:, k] * (1 - 1 / f)
    elif kind == "outside":   # a start outside, on a face or on an edge
        la[:, 1] = np.where(rng.random(n) < 0.5, 0.0, -2.0 ** rng.uniform(-60, 1, n))
        la[:, 2] = np.where(rng.random(n) < 0.3, 0.0, la[:, 2])
        la[:, 3] = np.where(rng.random(n) < 0.1, -0.0, la[:, 3])
    elif kind == "tiny":      # down to subnormals, starts and ends of any two sizes
        la = rng.random((n, 4)) * 2.0 ** rng.uniform(-160, 0, (n, 4)) * (rng.random((n, 4)) < 0.8)
        lb = rng.choice([-1.0, -1.0, 1.0], (n, 4)) * rng.random((n, 4)) * 2.0 ** rng.uniform(-160, 0, (n, 4))
    elif kind == "huge":      # past the FP32 range, infinities, NaN
        lb = lb * 2.0 ** rng.uniform(60, 300, (n, 4))
        lb[rng.random((n, 4)) < 0.05] = -np.inf
        lb[rng.random((n, 4)) < 0.05] = np.nan
    return np.ascontiguousarray(la), np.ascontiguousarray(lb)


@pytest.mark.parametrize("off", [-2, 0, 2])
@pytest.mark.parametrize("kind", ["plain", "ties", "outside", "tiny", "huge"])
def test_exit_face(lib, kind, off):
    la, lb = _pieces(kind)
    n = len(la)
    entry = np.random.default_rng(7).integers(-1, 4, n).astype(np.int32)
    kx, s = np.empty(n, np.int32), np.empty(n)
    lib.set_off(off)
    lib.t_exit(C.c_int64(n), *(a.ctypes.data_as(C.c_void_p) for a in (la, lb, entry, kx, s)))
    lib.set_off(0)
    with np.errstate(all="ignore"):
        sk = la / (la - lb)
        sk = np.where(sk < 0.0, 0.0, sk)
        sk = np.where((lb < 0.0) & (np.arange(4) != entry[:, None]) & ~np.isnan(sk), sk, np.inf)
    want = np.where(np.isinf(sk).all(1), -1, np.argmin(sk, 1))   # the lowest face on ties
    assert np.array_equal(kx, want)
    assert np.array_equal(s, sk.min(1))
    assert (want >= 0).sum() > n // 4
