"""A kernel chosen for a handle with the dissipation term or a density ratio is
the kernel that runs, and what is reported: left alone the pass after the
pre-pass (a part of 128 cells per CTA), chosen another tile shape or grid the
step that computes all again.  States do not change with an FP64 choice (the
operations are the same), nor with the FP32 choice of kernel 0's grid."""
import pytest

from paper_1412_6238_gb300 import workloads as wl
from paper_1412_6238_gb300.lbe import LBE

pytestmark = pytest.mark.gpu


def handle(storage, nx, ny, **options):
    w = wl.droplet(nx, ny, 20.0, nx / 2.0, ny / 2.0, Re=0.2, Ma=10.0, Ca=0.05, eta_m=0.2,
                   eta_r=0.5, lam_r=0.5)
    w.params.update(options)
    return LBE(w, storage=storage)


def tiles(nx, ny, tx, ty):
    return -(-nx // tx) * -(-ny // ty)


@pytest.mark.parametrize("storage,options,pre,parts", [
    ("f32", dict(dissip=1), (32, 8), 2), ("f64", dict(dissip=1), (16, 8), 1),
    ("f64", dict(rho2=3.0, dissip=1), (16, 8), 1), ("f64", dict(rho2=0.5), (16, 8), 1)])
def test_the_choice_runs(storage, options, pre, parts):
    import torch
    nx, ny = 203, 97
    a = handle(storage, nx, ny, **options)
    n = parts * tiles(nx, ny, *pre)
    assert a.get_tile() == dict(kernel=0, grid=n, seg_rows=0, items=n)
    b = handle(storage, nx, ny, **options)
    b.set_tile(0, -1)
    assert b.get_tile()["items"] == b.get_tile()["grid"] == tiles(nx, ny, *pre)
    for s in (a, b):
        s.step(9)
    assert torch.equal(a.get_state(), b.get_state())
    b.set_tile(0)  # and back, with the steps before and after in either way
    assert b.get_tile() == a.get_tile()
    a.set_tile(0, 7)
    assert a.get_tile()["grid"] == 7
    for s in (a, b):
        s.step(70)
    assert torch.equal(a.get_state(), b.get_state())
    if storage == "f32":
        for kernel, shape in ((1, (64, 4)), (2, (32, 16)), (3, (64, 8)), (4, (128, 4))):
            a.set_tile(kernel)
            assert a.get_tile()["kernel"] == kernel
            assert a.get_tile()["items"] == tiles(nx, ny, *shape)
