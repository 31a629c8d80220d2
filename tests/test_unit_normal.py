"""The unit normal of the FP32 reverse sweep, formed in two floats, against FP64:
the exact normal rounded to FP32, half a unit in the last place and 2^-12 of one
for the 2^-36 (2^-40 of each of some sixteen roundings) it may be off, and 2^-44
of the differences of c whose sum the gradient is.  Fields: an interface, its far
sides where c is all but uniform, noise in the low parts, gradients around and
far below eta_n, and none at all."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1412_6238_gb300", "csrc")
SOURCE = r'''
#include "lbe_two.cuh"
extern "C" void normals(const float* c, const float* cl, int nx, int ny, float eh, float el,
                        float* ox, float* oy) {
  for (int y = 1; y < ny - 1; y++)
    for (int x = 1; x < nx - 1; x++)
      lbe::unit_normal(c, cl, y * nx + x, nx, lbe::Two{eh, el}, ox[y * nx + x], oy[y * nx + x]);
}
'''


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("normal")
    (d / "n.cpp").write_text(SOURCE)
    so = str(d / "n.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC",
                    "-I" + CSRC, "-o", so, str(d / "n.cpp")], check=True)
    return ctypes.CDLL(so)


@pytest.mark.parametrize("eta_n", [1e-8, 1e-6, 3e-3, 0.5])
@pytest.mark.parametrize("noise", [0.0, 1e-12, 1e-7, 1e-3])
def test_rounded_once(lib, eta_n, noise):
    nx, ny = 160, 120
    rng = np.random.default_rng(2)
    y, x = np.mgrid[0:ny, 0:nx]
    c = 0.5 - 0.5 * np.tanh((np.hypot(x - 70.3, y - 55.7) - 30.0) / 1.5)
    c = c + noise * rng.standard_normal(c.shape)
    c[:20, :20] = 0.25
    hi = c.astype(np.float32)
    lo = (c - hi).astype(np.float32)
    c = hi.astype(np.float64) + lo
    e = 144.0 * eta_n * eta_n
    eh = np.float32(e)
    el = np.float32(e - float(eh))
    ox, oy = np.zeros_like(hi), np.zeros_like(hi)
    p = lambda a: a.ctypes.data_as(ctypes.c_void_p)  # noqa: E731
    lib.normals(p(hi), p(lo), nx, ny, ctypes.c_float(eh), ctypes.c_float(el),
                p(ox), p(oy))
    E, W, N, S = c[1:-1, 2:], c[1:-1, :-2], c[2:, 1:-1], c[:-2, 1:-1]
    d1, d2 = c[2:, 2:] - c[:-2, :-2], c[:-2, 2:] - c[2:, :-2]
    gx, gy = (4 * (E - W) + (d1 + d2)) / 12, (4 * (N - S) + (d1 - d2)) / 12
    s = np.sqrt(gx * gx + gy * gy + eta_n * eta_n)
    terms = (4 * np.maximum(abs(E - W), abs(N - S)) + abs(d1) + abs(d2)) / 12 / s
    for got, want in ((ox, gx / s), (oy, gy / s)):
        got = got[1:-1, 1:-1]
        assert np.isfinite(got).all()
        ulp = np.spacing(np.abs(want).astype(np.float32)).astype(np.float64)
        # (2^-100: where products leave FP32's range)
        bound = ulp * (0.5 + 2.0**-12) + terms * 2.0**-44 + 2.0**-100
        assert (np.abs(got - want) <= bound).all()
