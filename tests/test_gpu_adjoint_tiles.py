"""The tiled adjoint kernels (32 x 8 cells per block) where tiles can go wrong:
grids smaller than a tile, partial tiles, a top wall one row into a tile (row
ny then lies two rows above the tile below), one-column and two-row grids.

FP64: <a_out, V> of one adjoint step along random directions against the
central difference of the oracle's step.  eta_n = 1e-2 keeps the normal smooth
at the scale of h = 1e-7: the truncation error, of relative size (h / eta_n)^2
= 1e-10, and the rounding of J, 1e-16 sqrt(27 N) / h relative to a difference
of size sqrt(27 N), 1e-9, both stay below the bound 1e-6.

FP32: the gradient of a short run against the FP64 handle's.  Every FP32
product is off by 1e-7 and the smooth normal amplifies by at most 1 / eta_n:
1e-5, against the bound 1e-4."""
import dataclasses

import numpy as np
import pytest

from paper_1412_6238_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SIZES = [(1, 2), (2, 3), (5, 9), (31, 8), (33, 10), (40, 17), (64, 25), (70, 16)]


def _case(nx, ny):
    rng = np.random.default_rng(nx * 100 + ny)
    w = W.droplet(nx, ny, max(2.0, min(nx, ny) / 3.0), nx / 2.0, ny / 2.0 - 0.3, Re=0.1, Ma=10.0,
                  Ca=0.05, eta_m=0.2, eta_r=0.5, lam_r=2.0,
                  dT0=rng.normal(0.0, 1e-3, size=(ny, nx)))
    return dataclasses.replace(w, params=dict(w.params, eta_n=1e-2, ay=-2e-5))


def _lbe():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_6238_gb300.lbe import LBE
    return torch, LBE


@pytest.mark.parametrize("nx,ny", SIZES)
def test_adjoint_step_directions(orc, nx, ny):
    torch, LBE = _lbe()
    w = _case(nx, ny)
    Q = orc.run(w.params, orc.init(w.params, w.c0, w.T0, w.Tbot, w.Ttop), w.Tbot, w.Ttop, 4)
    rng = np.random.default_rng(3)
    a = rng.standard_normal(Q.shape)
    sim = LBE(w, storage="f64")
    out, _ = sim.adjoint_step(torch.from_numpy(Q).cuda(), torch.from_numpy(a).cuda(), 0.0)
    out = out.cpu().numpy()
    sim.close()
    h = 1e-7

    def J(q):
        return float((a * orc.run(w.params, q, w.Tbot, w.Ttop, 1)).sum())

    for planes in (slice(0, 9), slice(9, 18), slice(18, 27)):
        V = np.zeros_like(Q)
        V[planes] = rng.standard_normal(V[planes].shape)
        fd = (J(Q + h * V) - J(Q - h * V)) / (2 * h)
        ad = float((out * V).sum())
        scale = np.linalg.norm(out[planes]) * np.linalg.norm(V)
        assert abs(ad - fd) <= 1e-6 * scale, (planes, ad, fd)


@pytest.mark.parametrize("storage", ["f32", "f16mix", "f16dev", "bf16dev"])
@pytest.mark.parametrize("nx,ny", [(5, 9), (33, 10), (40, 17)])
def test_gradient_fp32(storage, nx, ny):
    _, LBE = _lbe()
    w = _case(nx, ny)
    # (the 16-bit storages hold the trajectory to 2^-11 or, BF16, 2^-8 of the
    # deviations, amplified as above by what divides by eta_n)
    tol = {"f32": 1e-4, "f16mix": 2e-2, "f16dev": 2e-2, "bf16dev": 1e-1}[storage]
    r = {}
    for st in ("f64", storage):
        sim = LBE(w, storage=st)
        r[st] = sim.adjoint(6, 3, 4, want_dQ0=True)
        sim.close()
    for key in ("dT0", "dQ0"):
        a, b = r["f64"][key], r[storage][key]
        assert float((a - b).norm()) <= tol * float(a.norm()), key
