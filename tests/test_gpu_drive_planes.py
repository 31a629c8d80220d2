"""A varying density or the dissipation term: the step whose pre-pass leaves all
it computes to the pass that collides, against the step that computes it again
(which a batch with a plain instance takes).  The operations are the same.
FP64, compiled without contraction: the same bits.  FP32, where a product and a
sum may be contracted in one kernel and not in the other: over four steps, each
with at most 8 roundings of 6e-8 in a population, 2e-6 of its plane's largest
value."""
import numpy as np
import pytest

from paper_1412_6238_gb300 import workloads as wl
from paper_1412_6238_gb300.lbe import LBE

pytestmark = pytest.mark.gpu


def drop(nx, ny, **options):
    w = wl.droplet(nx, ny, max(2.0, min(nx, ny) / 4.0), nx / 2.0, ny / 2.0, Re=0.2, Ma=10.0,
                   Ca=0.05, eta_m=0.2, eta_r=0.5, lam_r=0.5)
    w.params.update(options)
    return w


@pytest.mark.parametrize("storage,sizes,options", [
    ("f64", [(130, 100)], dict(rho2=3.0)),
    ("f64", [(97, 131)], dict(dissip=1)),
    ("f64", [(150, 83), (3, 9)], dict(rho2=0.5, dissip=1, cos_wet=0.3)),
    ("f64", [(10, 1200)], dict(rho2=2.0, interp=1, wall_mid=1)),
    ("f32", [(1, 2)], dict(dissip=1)),
    ("f32", [(33, 17)], dict(dissip=1)),
    ("f32", [(32, 8), (95, 41)], dict(dissip=1, interp=1, wall_mid=1, cos_wet=0.3)),
])
def test_planes_or_again(storage, sizes, options):
    ws = [drop(nx, ny, **options) for nx, ny in sizes]
    planes = LBE(ws, storage=storage)
    again = LBE(ws + [drop(120, 100)], storage=storage)
    planes.step(4)
    again.step(4)
    for j in range(len(ws)):
        a, b = planes.get_state(j).numpy(), again.get_state(j).numpy()
        if storage == "f64":
            assert np.array_equal(a, b)
        else:
            s = np.abs(b).max(axis=(1, 2), keepdims=True)
            assert (np.abs(a - b) <= 2e-6 * s).all()
