"""The device memory an FP64 gradient may take: 27 planes for each of a segment's
k + 1 states and 99 planes besides (as the first version took), the checkpoints
and a quarter of a GB for what the driver rounds up.  With no more than that
free the call must succeed."""
import pytest

from paper_1412_6238_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def test_a_segment_fits():
    torch = pytest.importorskip("torch")
    from paper_1412_6238_gb300.lbe import LBE
    nx, ny, k = 384, 320, 300
    w = wl.droplet(nx, ny, 40.0, nx / 2.0, ny / 2.0, Re=1.0, Ma=10.0, Ca=0.05, eta_m=0.2,
                   eta_r=0.5, lam_r=0.5)
    sim = LBE(w, storage="f64")
    sim.adjoint(2, 1, 1)  # (modules and workspaces are there)
    need = (27 * (k + 1) + 99) * 8 * nx * ny + 2 * sim.state_bytes + (1 << 28)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    free, _ = torch.cuda.mem_get_info()
    assert free > need
    hold = torch.empty(free - need, dtype=torch.uint8, device="cuda")
    try:
        r = sim.adjoint(k, 1, k)
    finally:
        del hold
        torch.cuda.empty_cache()
    assert r["loss"] == r["loss"]
    sim.close()
