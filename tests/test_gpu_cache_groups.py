"""The node cache of the multistep split with a group of lanes per marker,
against the FP64 oracle where entries are kept and replaced side by side in
one warp: markers at rest beside markers that cross cells in every sub-step,
and bond counts from none to all partners, so the groups of a warp run at
different speeds.  A lane that took a replaced entry for its own would read
the node of another cell.  Bounds as in test_gpu_coupling (FP64 storage:
roundoff)."""
import numpy as np
import pytest

import synth
from oracle import coupling as OC
from tests.gpu_helpers import make_pair, rel_l2, require_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M", [3, 13, 64])
@pytest.mark.parametrize("n", [1, 3])
@pytest.mark.parametrize("walls", [False, True])
def test_cached_nodes_of_crossing_markers_match_oracle(M, n, walls):
    require_cuda()
    shape = (12, 14, 16)
    nz, ny, nx = shape
    rng = np.random.default_rng(100 * n + M)
    pos = rng.uniform(0.0, 1.0, (M, 3)) * [nx, ny, nz - 4.0] + [0.0, 0.0, 2.0]
    vel = 0.3 * rng.choice([-1.0, 0.0, 1.0], (M, 3))
    vel[:, 2] *= 0.5                       # (four steps: clear of the walls)
    # marker 0 is bonded to every third one, the others of those in a chain
    third = np.arange(3, M, 3)
    bonds = np.array([(0, j) for j in third] + [(j, j + 1) for j in third if j + 1 < M])
    parts = dict(pos=pos, vel=vel, mass=np.full(M, 30.0))
    if len(bonds):
        parts.update(bonds=bonds, bond_k=0.02, bond_r0=2.0)
    fbar0 = synth.random_populations(shape, seed=8, amp=1e-3)
    box, sm = make_pair(shape, fbar0, coll="mrt", tau=0.8, walls=walls, storage="f64", kind="fc",
                        stencil="trilinear", gamma=0.3, split="inside", n=n, parts=parts)
    for _ in range(4):
        box.step(1)
        sm.step()
        pos_g, vel_g, fh = box.get_particles()
        assert np.abs(OC.min_image(pos_g - sm.parts.pos, shape, walls)).max() < 1e-11
        assert np.abs(vel_g - sm.parts.vel).max() < 1e-11
        assert np.abs(fh - sm.last_Fh).max() < 1e-11
    _, u = box.get_fields()
    assert rel_l2(u, sm.fluid_velocity()) < 1e-10
    assert box.check() == 0
    box.close()
