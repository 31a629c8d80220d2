"""Where and how fields may go: device buffers the kernel writes itself, in
both types, all or some of them; and the ones that are copied to, at an address
no double can be stored at, overlapping (written in order: the last one stays)
and on the host.  All hold the same values: FP32 is the FP64 value rounded."""
import ctypes

import numpy as np
import pytest
import torch

from helpers import gpu_fields, oracle_fields
from paper_1412_6238_gb300 import workloads as wl
from paper_1412_6238_gb300.lbe import FIELD_NAMES, LBE

pytestmark = pytest.mark.gpu


def export(sim, ptrs, on_device, dtype):
    a = (ctypes.c_void_p * 5)(*ptrs)
    mask = sum(1 << k for k in range(5) if ptrs[k])
    sim._check(sim._L.lbe_fields(sim._h, 0, mask, a, on_device, dtype))


@pytest.mark.parametrize("storage,nx,ny", [("f64", 33, 18), ("f32", 131, 20), ("f16mix", 4, 9),
                                           ("f16dev", 32, 8), ("bf16dev", 65, 33)])
def test_outputs_hold_the_same_values(storage, nx, ny):
    w = wl.droplet(nx, ny, 4.0, nx / 2.0, ny / 2.0, Re=0.2, Ma=10.0, Ca=0.05, eta_m=0.2,
                   eta_r=0.5, lam_r=0.5)
    sim = LBE(w, storage=storage)
    sim.step(5)
    N = nx * ny
    ref = sim.fields(device="cpu")
    full = torch.stack([ref[k].reshape(-1) for k in FIELD_NAMES])
    for dtype, code, size in ((torch.float64, 0, 8), (torch.float32, 1, 4)):
        want = full.to(dtype)
        for device in ("cuda", "cpu"):
            buf = torch.full((5, N), -7.0, dtype=dtype, device=device)
            export(sim, [buf[k].data_ptr() for k in range(5)], device == "cuda", code)
            assert torch.equal(buf.cpu(), want)
            buf.fill_(-7.0)
            export(sim, [0, buf[1].data_ptr(), 0, 0, buf[4].data_ptr()], device == "cuda", code)
            assert torch.equal(buf[[1, 4]].cpu(), want[[1, 4]])
            assert (buf[[0, 2, 3]] == -7.0).all()
            # one buffer for all, and each one cell on from the one before
            export(sim, [buf[0].data_ptr()] * 5, device == "cuda", code)
            assert torch.equal(buf[0].cpu(), want[4])
            flat = torch.zeros(N + 4, dtype=dtype, device=device)
            export(sim, [flat.data_ptr() + size * k for k in range(5)], device == "cuda", code)
            assert torch.equal(flat[:4].cpu(), want[:4, 0])
            assert torch.equal(flat[4:].cpu(), want[4])
    # doubles at an address that is a multiple of four only
    raw = torch.zeros(2 * N + 1, dtype=torch.float32, device="cuda")
    export(sim, [raw.data_ptr() + 4, 0, 0, 0, 0], True, 0)
    assert torch.equal(raw[1:].cpu().view(torch.float64), full[0])


@pytest.mark.parametrize("options", [{}, dict(interp=1, wall_mid=1, cos_wet=0.4)])
@pytest.mark.parametrize("storage", ["f32", "f16mix", "f16dev", "bf16dev"])
@pytest.mark.parametrize("nx,ny", [(3, 8), (4, 2), (5, 9), (127, 11), (128, 3), (129, 40),
                                   (300, 97)])
def test_fields_are_those_of_the_state(orc, storage, nx, ny, options):
    """The fields of a single-precision storage against the oracle's of the same populations.  FP32 sums of nine
    terms: at most 8 roundings of 6e-8 of the largest, 5e-7; c, p, T to 2e-6 of
    their largest value.  u holds half the force, whose curvature comes from
    differences of c near 1e-2 of it: 1e-4 of the largest |u|."""
    def drop(nx, ny):
        w = wl.droplet(nx, ny, max(2.0, min(nx, ny) / 4.0), nx / 2.0, ny / 2.0, Re=0.2, Ma=10.0,
                       Ca=0.05, eta_m=0.2, eta_r=0.5, lam_r=0.5)
        w.params.update(options)
        return w
    w = drop(nx, ny)
    sim = LBE([drop(33, 12), w], storage=storage)
    sim.step(6)
    got = gpu_fields(sim, 1)
    want = oracle_fields(orc, w, sim.get_state(1).numpy())
    u = max(np.abs(want["ux"]).max(), np.abs(want["uy"]).max())
    for k in FIELD_NAMES:
        scale, tol = (u, 1e-4) if k in ("ux", "uy") else (np.abs(want[k]).max(), 2e-6)
        assert np.abs(got[k] - want[k]).max() <= tol * scale, k


@pytest.mark.parametrize("nx,ny,options", [(4, 524299, {}), (2051, 1031, {}),
                                           (131, 16103, dict(interp=1, wall_mid=1, cos_wet=0.4))])
@pytest.mark.parametrize("storage", ["f32", "f16mix", "f16dev", "bf16dev"])
def test_fields_of_large_grids(orc, storage, nx, ny, options):
    """The same, with drops of the same sizes and the same bounds, from the number
    of cells on where the strip kernel writes the fields (sigma varying from wall
    to wall as in a grid of 20 rows)."""
    assert nx * ny >= 1 << 21
    w = wl.droplet(nx, ny, max(2.0, min(nx, 40) / 4.0), nx / 2.0, ny / 2.0, Re=0.2, Ma=10.0,
                   Ca=0.05, eta_m=0.2, eta_r=0.5, lam_r=0.5)
    w.params.update(options, sigmaT=w.params["sigmaT"] * 20 / ny)
    sim = LBE([w], storage=storage)
    sim.step(6)
    got = gpu_fields(sim, 0)
    want = oracle_fields(orc, w, sim.get_state(0).numpy())
    u = max(np.abs(want["ux"]).max(), np.abs(want["uy"]).max())
    for k in FIELD_NAMES:
        scale, tol = (u, 1e-4) if k in ("ux", "uy") else (np.abs(want[k]).max(), 2e-6)
        assert np.abs(got[k] - want[k]).max() <= tol * scale, k
