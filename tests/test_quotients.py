"""The FP64 quotients of the step, compiled for the host, against the division:
equal bit for bit.  Divisors of every kind (1, 1/3, reciprocals within and beyond
a quarter of their last place, and those outside 2^-60 .. 2^60, of a constant
and of a cell, negative ones too); numerators with random mantissas, with runs of
zeros and ones at either end, next to multiples of the divisor, and at the edges:
zeros, subnormals, 2^-900, 2^900, infinities, NaN."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1412_6238_gb300", "csrc")
SOURCE = r"""
#include "lbe_quot.cuh"
using namespace lbe;
// kind of b: a constant's (cell = 0) or a cell's; q[i] = a[i] / b as the step forms it
extern "C" int quotients(const double* a, double* q, long n, double b, int cell) {
  const double y = 1.0 / b;
  const Den<double> d{b, y, cell ? cell_kind(b) : constant_kind(b, y)};
  for (long i = 0; i < n; i++) q[i] = dv(a[i], d);
  return d.kind;
}
extern "C" void thirds(const double* a, double* q, long n) {
  for (long i = 0; i < n; i++) q[i] = dv_cs2(a[i]);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("quot")
    (d / "q.cpp").write_text(SOURCE)
    so = str(d / "q.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC",
                    "-I" + CSRC, "-o", so, str(d / "q.cpp")], check=True)
    return ctypes.CDLL(so)


def _mantissas(rng, n):
    m = rng.integers(0, 1 << 52, n)
    k = rng.integers(0, 53, n)
    ends = [m, (1 << 52) - 1 - (m >> k), m >> k, (m >> k) << k & (1 << 52) - 1]
    return 1.0 + np.concatenate(ends) / 2.0**52


def numerators(b, seed=0, n=20000):
    rng = np.random.default_rng(seed)
    m = _mantissas(rng, n)
    a = np.ldexp(m, rng.integers(-60, 60, m.size))
    wide = np.ldexp(m, rng.integers(-1074, 1024, m.size))
    with np.errstate(all="ignore"):
        # next to a multiple of b, and to the middle between two quotients
        near = [a * b, np.nextafter(a * b, 0), np.nextafter(a * b, np.inf),
                np.nextafter(a * b * (1 + 2.0**-53), np.inf)]
    edge = np.array([0.0, 5e-324, 1e-310, 2.0**-1022, 2.0**-901, 2.0**-900, 2.0**900, 2.0**901,
                     1.7e308, np.inf, np.nan])
    edge = np.concatenate([edge, np.nextafter(edge, 0), np.nextafter(edge, np.inf)])
    a = np.concatenate([a, wide, edge] + near)
    return np.concatenate([a, -a])


def divisors():
    rng = np.random.default_rng(5)
    d = [1.0, 1.0 / 3.0, 3.0, 0.9, 1.1, 1.7, 4.0 / 9.0, 0.7 / 3.0, 1.3 * 1.7 / 3.0, 2.0**-60,
         np.nextafter(2.0**60, 0), 1.0 + 2.0**-52, 2.0 - 2.0**-52]
    d += list(_mantissas(rng, 3) * np.ldexp(1.0, rng.integers(-50, 50, 12)))
    return [float(x) for x in d]


OUTSIDE = [2.0**-61 * 1.7, 2.0**60, 1e-200, 1e200, 1e-305, 5e-324, 1.7e308]


def check(lib, b, cell):
    a = numerators(b)
    q = np.empty_like(a)
    p = lambda v: v.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    kind = lib.quotients(p(a), p(q), ctypes.c_long(a.size), ctypes.c_double(b), cell)
    with np.errstate(all="ignore"):
        want = a / b
    same = (q.view(np.int64) == want.view(np.int64)) | (np.isnan(q) & np.isnan(want))
    assert same.all(), (kind, a[~same][:3], q[~same][:3], want[~same][:3])
    return kind


@pytest.mark.parametrize("b", divisors())
def test_constants(lib, b):
    assert check(lib, b, 0) in (0, 1, 2, 4)


@pytest.mark.parametrize("b", divisors() + [-x for x in divisors()])
def test_cells(lib, b):
    assert check(lib, b, 1) == 2


@pytest.mark.parametrize("b", OUTSIDE + [-x for x in OUTSIDE] + [0.0, -0.0, np.inf, np.nan])
def test_outside(lib, b):
    assert check(lib, b, 1) == 3
    if b > 0 and np.isfinite(b):
        assert check(lib, b, 0) == 3


def test_thirds(lib):
    rng = np.random.default_rng(9)
    near = np.concatenate([
        np.ldexp(x + k * 2.0**-52, e) for x in (1.0, 4.0 / 3.0, 5.0 / 3.0, 2.0)
        for e in (-300, 0, 17) for k in (np.arange(-20000, 20000), rng.integers(-2**30, 2**30, 20000))])
    a = np.concatenate([numerators(1.0 / 3.0, 3, 200000), near])
    q = np.empty_like(a)
    p = lambda v: v.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    lib.thirds(p(a), p(q), ctypes.c_long(a.size))
    with np.errstate(all="ignore"):
        want = a / (1.0 / 3.0)
    assert ((q.view(np.int64) == want.view(np.int64)) | (np.isnan(q) & np.isnan(want))).all()
