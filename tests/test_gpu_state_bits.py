"""The bits of states.  How a multiplication and an addition round together is
the compiler's choice wherever a kernel does not fix it, and in the 16-bit
storages a value next to a tie is then stored the other way: a run continued
under another build would part from its own past.  The digests are of states
made before the kernels read their constants from shared memory and before the
FP64 quotients were rewritten; inputs are built from whole numbers, so that no library function enters.  The wide grid is
all walls and strip edges, the other one mostly bulk."""
import hashlib
import json
import os

import numpy as np
import pytest

from paper_1412_6238_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

VARIANTS = dict(interp=1, wall_mid=1, cos_wet=0.375)
OPTIONS = {"plain": {}, "variants": VARIANTS, "dissipation": dict(dissip=1),
           "dissipation variants": dict(dissip=1, **VARIANTS)}
GRIDS = [(30001, 6), (300, 97)]
GOLDEN = os.path.join(os.path.dirname(__file__), "golden", "state_bits.json")


def cases():
    for storage in ("f32", "f16mix", "f16dev", "bf16dev"):
        for options in ("plain", "variants"):
            for nx, ny in GRIDS:
                for kernel in (0, 1, 2, 3, 4, 7, 8):
                    yield storage, options, nx, ny, kernel
    for options in ("dissipation", "dissipation variants"):
        for nx, ny in GRIDS:
            for kernel in range(5):
                yield "f32", options, nx, ny, kernel


def digest(storage, options, nx, ny, kernel, batched=False):
    """Digest of the populations after 12 steps from an FP64 state, of the
    instance alone or beside one without options."""
    from paper_1412_6238_gb300.lbe import LBE
    w = wl.droplet(nx, ny, 4.0, 8.0, 3.0, Re=0.05, Ma=10.0, Ca=0.05, eta_m=0.2, eta_r=0.5,
                   lam_r=0.5)
    w.params.update({k: float("%.9g" % v) for k, v in w.params.items() if isinstance(v, float)})
    w.params.update(OPTIONS[options])
    rng = np.random.default_rng(11)

    def whole(lo, hi, *size):
        return rng.integers(lo, hi, size=size) / 2.0**20
    w.c0[:] = whole(0, 300000, ny, nx) + (np.arange(nx) // 40 % 2) * 0.625
    w.Tbot[:] = 1.0625 + whole(0, 20000, nx)
    w.Ttop[:] = 0.9375 + whole(0, 20000, nx)
    w.T0[:] = 1.0 + whole(-2000, 2000, ny, nx)
    ref = LBE(w, storage="f64")
    ref.step(10)
    Q = ref.get_state()
    ref.close()
    plain = wl.droplet(70, 33, 8.0, 30.0, 16.0, Re=0.2, Ma=10.0, Ca=0.05, eta_m=0.2, eta_r=0.5,
                       lam_r=0.5)
    sim = LBE([w, plain] if batched else w, storage=storage)
    sim.set_tile(kernel)
    sim.set_state(Q)
    sim.step(1)
    sim.step(11)
    out = sim.get_state().cpu().numpy()
    sim.close()
    assert np.isfinite(out).all()
    return hashlib.sha256(np.ascontiguousarray(out).tobytes()).hexdigest()[:16]


def golden(storage, options, nx, ny, kernel):
    with open(GOLDEN) as f:
        return json.load(f)["%s %s %dx%d kernel %d" % (storage, options, nx, ny, kernel)]


@pytest.mark.parametrize("storage,options,nx,ny,kernel", list(cases()))
def test_state_bits(storage, options, nx, ny, kernel):
    assert digest(storage, options, nx, ny, kernel) == golden(storage, options, nx, ny, kernel)


@pytest.mark.parametrize("options", ["dissipation", "dissipation variants"])
@pytest.mark.parametrize("nx,ny", GRIDS)
def test_dissipation_in_any_company(options, nx, ny):
    """Beside a plain instance the step computes again what the pre-pass leaves
    in planes otherwise (or where memory has no room for them)."""
    assert digest("f32", options, nx, ny, 0, batched=True) == golden("f32", options, nx, ny, 0)
