"""The 4- and 3-point interpolation of few markers without the node-moment
field (populations pulled, several nodes in flight) against the FP64 oracle,
and against the same box with the field (same bits in every storage): one
marker, a partial last warp, markers at both walls and across the periodic
faces.  Bounds as in test_gpu_coupling (FP64 storage: roundoff)."""
import numpy as np
import pytest

import synth
from oracle import coupling as OC
from tests.gpu_helpers import make_pair, rel_l2, require_cuda

pytestmark = pytest.mark.gpu


def _pair(stencil, kind, M, walls, storage):
    shape = (11, 10, 13)
    nz, ny, nx = shape
    rng = np.random.default_rng(M)
    pos = rng.uniform(0.0, 1.0, (M, 3)) * [nx, ny, nz]
    if walls:
        pos[:, 2] = rng.uniform(0.2, nz - 1.2, M)
    parts = dict(pos=pos)
    if kind != "ibm":
        parts.update(vel=0.02 * rng.standard_normal((M, 3)), mass=2.0)
    if M > 1:
        bonds = np.stack([np.arange(M - 1), np.arange(1, M)], axis=1)[::3]
        parts.update(bonds=bonds, bond_k=0.002, bond_r0=2.0)
    fbar0 = synth.random_populations(shape, seed=4, amp=1e-3)
    return shape, make_pair(shape, fbar0, coll="mrt", tau=0.8, g=(1e-5, 0, 0), walls=walls,
                            storage=storage, kind=kind, stencil=stencil, gamma=0.3, parts=parts)


@pytest.mark.parametrize("stencil", ["peskin4", "peskin3"])
@pytest.mark.parametrize("kind", ["fc", "ibm"])
@pytest.mark.parametrize("M", [1, 45])
@pytest.mark.parametrize("walls", [False, True])
def test_pulled_nodes_match_oracle(stencil, kind, M, walls):
    require_cuda()
    from paper_1406_2211_gb300 import lbc
    shape, (box, sm) = _pair(stencil, kind, M, walls, "f64")
    box.set_option(lbc.LBC_OPT_NODE_MOMENTS, 0)
    box.step(3)
    for _ in range(3):
        sm.step()
    pos, vel, fh = box.get_particles()
    assert np.abs(OC.min_image(pos - sm.parts.pos, shape, walls)).max() < 1e-11
    if kind != "ibm":
        assert np.abs(vel - sm.parts.vel).max() < 1e-11
        assert np.abs(fh - sm.last_Fh).max() < 1e-11
    _, u = box.get_fields()
    assert rel_l2(u, sm.fluid_velocity()) < 1e-10
    assert box.check() == 0
    box.close()


@pytest.mark.parametrize("stencil", ["peskin4", "peskin3"])
@pytest.mark.parametrize("kind", ["fc", "ibm"])
@pytest.mark.parametrize("storage", ["f64", "f32", "f16dev", "bf16dev"])
@pytest.mark.parametrize("walls", [False, True])
def test_pulled_nodes_have_the_bits_of_the_field(stencil, kind, storage, walls):
    require_cuda()
    from paper_1406_2211_gb300 import lbc
    out = []
    for moments in (0, 1):
        _, (box, _) = _pair(stencil, kind, 45, walls, storage)
        box.set_option(lbc.LBC_OPT_NODE_MOMENTS, moments)
        box.step(4)
        out.append([box.get_populations(), *box.get_particles()])
        assert box.check() == 0
        box.close()
    for x, y in zip(*out):
        np.testing.assert_array_equal(x, y)
