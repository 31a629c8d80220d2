"""A run of many steps in one call (captured groups of steps, whose kernels
start before the one before them has ended) is bit for bit the run of as many
single steps, whatever the kernel, the storage and the place the count starts
at: the steps are the same operations, and the random bits of the stochastic
rounding depend on the step's number alone."""
import numpy as np
import pytest
import torch

from paper_1412_6238_gb300 import workloads as wl
from paper_1412_6238_gb300.lbe import LBE

pytestmark = pytest.mark.gpu


def drop(nx, ny, **options):
    w = wl.droplet(nx, ny, 5.0, nx / 2.0, ny / 2.0, Re=0.2, Ma=10.0, Ca=0.05, eta_m=0.2,
                   eta_r=0.5, lam_r=0.5)
    w.params.update(options)
    return w


# (4, 40): no wider than the ghost columns; (130, 33): a strip of 2 columns
@pytest.mark.parametrize("storage,kernel,nx,ny,options", [
    ("f64", 0, 5, 40, {}),
    ("f64", 0, 40, 33, dict(rho2=2.0)),
    ("f32", 0, 33, 40, dict(dissip=1)),
    ("f32", 7, 130, 33, {}),
    ("f32", 8, 130, 33, dict(cos_wet=0.3)),
    ("f32", 8, 256, 9, {}),
    ("f16mix", 0, 33, 40, {}),
    ("f16mix", 7, 4, 40, {}),
    ("f16mix", 8, 130, 33, {}),
    ("f16dev", 7, 130, 33, {}),
    ("f16dev", 8, 256, 9, {}),
    ("bf16dev", 8, 40, 33, {}),
])
def test_one_call_is_its_single_steps(storage, kernel, nx, ny, options):
    w = drop(nx, ny, **options)
    a, b = LBE(w, storage=storage), LBE(w, storage=storage)
    for s in (a, b):
        s.set_tile(kernel)
    # 67: groups of sixteen and three steps; 81 more from odd parity; 63, 2
    for n in (67, 81, 63, 2):
        a.step(n)
        for _ in range(n):
            b.step(1)
        assert torch.equal(a.get_state(), b.get_state())


def test_group_counts_its_steps(tmp_path):
    """A file saved within a run of groups goes on as the run does."""
    w = drop(64, 48)
    a = LBE(w, storage="f16mix")
    a.step(83)
    a.save(str(tmp_path / "s.lbe"))
    b = LBE(w, storage="f16mix")
    b.step(34)
    b.load(str(tmp_path / "s.lbe"))
    for s in (a, b):
        s.step(70)
    assert np.array_equal(a.get_state().numpy(), b.get_state().numpy())
