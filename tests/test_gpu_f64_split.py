"""The FP64 step of small grids, a tile's work divided among four warps, gives
the bits of the other FP64 tiles: an instance alone (few tiles) against the
same instance in a batch whose other one takes the batch to the 4 x 8 tile of
one warp (16 x 700) or to the 16 x 8 tile (130 x 100).  The operations on a cell
are the same in the same order, so nothing may differ."""
import pytest
import torch

from paper_1412_6238_gb300 import workloads as wl
from paper_1412_6238_gb300.lbe import LBE

pytestmark = pytest.mark.gpu


def drop(nx, ny, **options):
    w = wl.droplet(nx, ny, max(2.0, min(nx, ny) / 4.0), nx / 2.0, ny / 2.0, Re=0.2, Ma=10.0,
                   Ca=0.05, eta_m=0.2, eta_r=0.5, lam_r=0.5)
    w.params.update(options)
    return w


@pytest.mark.parametrize("options", [
    {}, dict(rho2=3.0), dict(dissip=1), dict(rho2=0.5, dissip=1),
    dict(interp=1, wall_mid=1, cos_wet=0.4, ax=1e-6)])
@pytest.mark.parametrize("nx,ny,other", [
    (1, 2, (16, 700)), (3, 7, (16, 700)), (4, 8, (130, 100)), (16, 101, (16, 700)),
    (17, 9, (130, 100)), (95, 97, (130, 100))])
def test_same_bits_as_the_other_tiles(nx, ny, other, options):
    w = drop(nx, ny, **options)
    alone, batch = LBE(w, storage="f64"), LBE([w, drop(*other)], storage="f64")
    for n in (1, 6):
        alone.step(n)
        batch.step(n)
        assert torch.equal(alone.get_state(0), batch.get_state(0))
