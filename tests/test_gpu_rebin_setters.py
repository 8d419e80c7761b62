"""Re-binning across a setter between single steps, against the FP64 oracle:
lbc_box_set_fields moves the step parity that numbers the re-binning flags, so
a re-sort requested by the step before it must still happen.  Markers cross
several tiles in the run; a lost request would leave them outside their bins
(LBC_ERR_STATE).  Bounds as in test_gpu_coupling (FP64 storage: roundoff).
"""
import numpy as np
import pytest

from oracle import coupling as OC
from oracle import lattice as OLat
from tests.gpu_helpers import make_pair, require_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("split,n", [("base", 1), ("inside", 2), ("outside", 2)])
def test_fields_set_after_every_step(split, n):
    require_cuda()
    shape = (16, 17, 18)
    rng = np.random.default_rng(5)
    M = 300                     # dense enough that some hit lists overflow into the search
    parts = dict(pos=rng.uniform(0.0, 1.0, (M, 3)) * [6.0, 6.0, 6.0] + 4.0,
                 vel=np.tile([0.23, 0.17, -0.21], (M, 1)), mass=np.full(M, 50.0))
    rho = np.ones(shape)
    u = np.zeros((3,) + shape)
    u[0] = 0.05
    feq = OLat.equilibrium(rho, u)
    box, sm = make_pair(shape, feq, tau=0.9, storage="f64", kind="fc", stencil="trilinear",
                        gamma=0.05, split=split, n=n, parts=parts)
    for _ in range(30):
        box.step(1)
        box.set_fields(rho, u)
        sm.step()
        sm.fbar = feq.copy()
        sm.Fa = np.zeros_like(u)
    assert box.check() == 0
    pos, vel, fh = box.get_particles()
    assert np.abs(OC.min_image(pos - sm.parts.pos, shape, False)).max() < 1e-11
    assert np.abs(vel - sm.parts.vel).max() < 1e-11
    assert np.abs(fh - sm.last_Fh).max() < 1e-11
    box.close()


@pytest.mark.parametrize("storage", ["f64", "f32", "f16dev"])
def test_markers_faster_than_a_cell_per_step(storage):
    """Base split: the binning keys are those of the force points, so markers
    of any speed stay inside their bins (here more than a cell per half step).
    FP32 and FP16: no error status, positions to the roundoff of velocities
    that a heavy marker hardly changes."""
    require_cuda()
    shape = (12, 13, 14)
    rng = np.random.default_rng(6)
    M = 40
    parts = dict(pos=rng.uniform(0.0, 1.0, (M, 3)) * [14.0, 13.0, 12.0],
                 vel=np.tile([2.3, -1.7, 2.1], (M, 1)), mass=np.full(M, 1e4))
    feq = OLat.equilibrium(np.ones(shape), np.zeros((3,) + shape))
    box, sm = make_pair(shape, feq, tau=0.9, storage=storage, kind="fc", stencil="trilinear",
                        gamma=1e-3, split="base", n=1, parts=parts)
    for _ in range(10):
        box.step(1)
        sm.step()
    assert box.check() == 0
    pos, vel, _ = box.get_particles()
    tol = 1e-11 if storage == "f64" else 1e-6
    assert np.abs(OC.min_image(pos - sm.parts.pos, shape, False)).max() < tol
    assert np.abs(vel - sm.parts.vel).max() < tol
    box.close()
