"""FP64 steps bitwise equal to the oracle where the quotients and the tile
shapes can go wrong: densities and heat capacities that take each way of
forming a quotient (divisor 1, 1/3, a rounded reciprocal within and beyond a
quarter of its last place), a density ratio, c down to the smallest subnormals
and exact zeros of both signs of u (where a remainder would underflow, the true
division), and widths on both sides of the narrow tile's limit (16)."""
import dataclasses

import numpy as np
import pytest

from paper_1412_6238_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(3, 8), (16, 9), (17, 25), (33, 17)])
@pytest.mark.parametrize("rho,cv,rho2", [(1.0, 1.0, 0.0), (0.9, 1.3, 0.0), (1.7, 0.7, 0.0),
                                         (1.1, 1.0, 3.3)])
def test_steps_bitwise(orc, nx, ny, rho, cv, rho2):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1412_6238_gb300.lbe import LBE
    w = W.droplet(nx, ny, max(2.0, min(nx, ny) / 3.0), nx / 2.0, ny / 2.0 - 0.3, Re=0.1, Ma=10.0,
                  Ca=0.05, eta_m=0.2, eta_r=0.5, lam_r=2.0)
    p = dict(w.params, rho=rho, cv=cv, ax=1e-6)
    if rho2:
        p["rho2"] = rho2
    c0 = w.c0.copy()
    # columns of tiny, subnormal and zero values of c off the drop
    for j, v in enumerate((1e-250, 1e-290, 1e-305, 5e-324, 0.0)):
        c0[j % ny, :] = v
    w = dataclasses.replace(w, params=p, c0=c0)
    sim = LBE(w, storage="f64")
    Q = orc.init(w.params, w.c0, w.T0, w.Tbot, w.Ttop)
    assert np.array_equal(sim.get_state().numpy(), Q) or rho2
    sim.set_state(Q)
    for n in (1, 2):
        sim.step(n)
        Q = orc.run(w.params, Q, w.Tbot, w.Ttop, n)
        got = sim.get_state().numpy()
        # a density ratio: hbar's wall values and the pre-pass differ in the
        # order of their operations from the oracle's (1e-13 elsewhere)
        if rho2:
            s = np.abs(Q).max(axis=(1, 2), keepdims=True)
            assert (np.abs(got - Q) <= 1e-13 * np.maximum(s, 1.0)).all()
        else:
            assert np.array_equal(got, Q)
    sim.close()
