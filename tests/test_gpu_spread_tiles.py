"""Trilinear spreading from the tiles' hit lists against the FP64 oracle where
a list can go wrong: axes of one tile, of a tile and one cell, of partial last
tiles and of two whole tiles (a stencil then meets a tile from both sides of
the periodic boundary), and so many markers that lists overflow into the
search.  Bounds as in test_gpu_coupling (FP64 storage: roundoff)."""
import numpy as np
import pytest

import synth
from oracle import coupling as OC
from tests.gpu_helpers import make_pair, rel_l2, require_cuda

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(4, 5, 7), (8, 6, 5), (9, 8, 4), (3, 20, 13), (16, 12, 8)])
@pytest.mark.parametrize("markers", [7, 500])
@pytest.mark.parametrize("walls", [False, True])
def test_hit_lists_match_oracle(shape, markers, walls):
    require_cuda()
    nz, ny, nx = shape
    rng = np.random.default_rng(7 + markers)
    pos = rng.uniform(0.0, 1.0, (markers, 3)) * [nx, ny, nz]
    if walls:
        pos[:, 2] = rng.uniform(-0.4, nz - 0.6, markers)
    pos[0] = [nx - 1.0, 0.0, 0.0]              # on nodes: zero weights drop the upper nodes
    parts = dict(pos=pos, vel=0.01 * rng.standard_normal((markers, 3)),
                 mass=np.full(markers, 2.0))
    fbar0 = synth.random_populations(shape, seed=9, amp=1e-3)
    # gamma small enough for many markers per cell (explicit in the others'
    # forces): gamma h M / N < 1
    box, sm = make_pair(shape, fbar0, tau=0.9, storage="f64", kind="fc", stencil="trilinear",
                        gamma=0.1, walls=walls, parts=parts)
    box.step(4)
    for _ in range(4):
        sm.step()
    p, v, fh = box.get_particles()
    assert np.abs(OC.min_image(p - sm.parts.pos, shape, walls)).max() < 1e-11
    assert np.abs(v - sm.parts.vel).max() < 1e-11
    assert np.abs(fh - sm.last_Fh).max() < 1e-11
    _, u = box.get_fields()
    assert rel_l2(u, sm.fluid_velocity()) < 1e-10
    assert box.check() == 0
    box.close()
