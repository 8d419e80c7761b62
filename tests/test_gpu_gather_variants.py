"""The trilinear interpolation's launch variants against the FP64 oracle at
the sizes where they change: eight lanes per marker (a partial last group and
a partial last warp, up to the marker count whose lanes fill the GPU), and
one lane per marker beyond it (populations pulled by the lane, or the node
cache of the multistep split, which a warp refills together).

Bounds as in test_gpu_coupling: FP64 storage computes every part in FP64, so
particles agree to 1e-11 and the fluid velocity to 1e-10 relative L2.
"""
import numpy as np
import pytest

import synth
from oracle import coupling as OC
from tests.gpu_helpers import make_pair, rel_l2, require_cuda

pytestmark = pytest.mark.gpu


def _resident():
    """Markers whose eight lanes are resident at once (96 per SM)."""
    import torch
    return 96 * torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("count", [1, 5, 8193, "resident", "resident+1"])
@pytest.mark.parametrize("split,n", [("base", 1), ("inside", 2)])
@pytest.mark.parametrize("walls", [False, True])
def test_trilinear_variants_match_oracle(count, split, n, walls):
    require_cuda()
    M = count if isinstance(count, int) else _resident() + (1 if count.endswith("+1") else 0)
    shape = (40, 44, 48) if M > 1000 else (11, 10, 13)
    nz, ny, nx = shape
    rng = np.random.default_rng(31 + M)
    pos = rng.uniform(0.0, 1.0, (M, 3)) * [nx, ny, nz]
    if walls:           # up to the walls: stencil nodes beyond them are dropped
        pos[:, 2] = rng.uniform(-0.4, nz - 0.6, M)
    parts = dict(pos=pos, vel=0.02 * rng.standard_normal((M, 3)), mass=rng.uniform(0.5, 2.0, M),
                 ext=1e-4 * rng.standard_normal((M, 3)))
    if M > 1:
        parts.update(bonds=np.stack([np.arange(M - 1), np.arange(1, M)], axis=1)[::3],
                     bond_k=0.01, bond_r0=1.0)
    fbar0 = synth.random_populations(shape, seed=4, amp=1e-3)
    box, sm = make_pair(shape, fbar0, coll="mrt", tau=0.8, g=(1e-5, 0, 0), walls=walls,
                        storage="f64", kind="fc", stencil="trilinear", gamma=0.5, split=split, n=n,
                        parts=parts)
    box.step(3)
    for _ in range(3):
        sm.step()
    pos, vel, fh = box.get_particles()
    assert np.abs(OC.min_image(pos - sm.parts.pos, shape, walls)).max() < 1e-11
    assert np.abs(vel - sm.parts.vel).max() < 1e-11
    assert np.abs(fh - sm.last_Fh).max() < 1e-11
    _, u = box.get_fields()
    assert rel_l2(u, sm.fluid_velocity()) < 1e-10
    assert box.check() == 0
    box.close()
