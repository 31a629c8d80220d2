"""Where and how fields may go on a grid large enough for the strip kernel to
write them: all or some, as doubles or floats (the double rounded), to the
device, the host, one buffer for all, overlapping buffers (written in order: the
last one stays) and an address no double can be stored at."""
import ctypes

import pytest
import torch

from paper_1412_6238_gb300 import workloads as wl
from paper_1412_6238_gb300.lbe import FIELD_NAMES, LBE

pytestmark = pytest.mark.gpu


def export(sim, ptrs, on_device, dtype):
    a = (ctypes.c_void_p * 5)(*ptrs)
    mask = sum(1 << k for k in range(5) if ptrs[k])
    sim._check(sim._L.lbe_fields(sim._h, 0, mask, a, on_device, dtype))


@pytest.mark.parametrize("storage", ["f32", "f16mix", "f16dev", "bf16dev"])
@pytest.mark.parametrize("nx,ny,options", [(2051, 1031, {}), (129, 16300, dict(cos_wet=0.4))])
def test_outputs_hold_the_same_values(storage, nx, ny, options):
    N = nx * ny
    assert N >= 1 << 21
    w = wl.droplet(nx, ny, 20.0, nx / 2.0, ny / 2.0, Re=0.2, Ma=10.0, Ca=0.05, eta_m=0.2,
                   eta_r=0.5, lam_r=0.5)
    w.params.update(options)
    sim = LBE(w, storage=storage)
    sim.step(5)
    ref = sim.fields(device="cpu")
    full = torch.stack([ref[k].reshape(-1).to(torch.float64) for k in FIELD_NAMES])
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
            export(sim, [buf[0].data_ptr()] * 5, device == "cuda", code)
            assert torch.equal(buf[0].cpu(), want[4])
            flat = torch.zeros(N + 4, dtype=dtype, device=device)
            export(sim, [flat.data_ptr() + size * k for k in range(5)], device == "cuda", code)
            assert torch.equal(flat[:4].cpu(), want[:4, 0])
            assert torch.equal(flat[4:].cpu(), want[4])
    raw = torch.zeros(2 * N + 1, dtype=torch.float32, device="cuda")
    export(sim, [raw.data_ptr() + 4, 0, 0, 0, 0], True, 0)
    assert torch.equal(raw[1:].cpu().view(torch.float64), full[0])
