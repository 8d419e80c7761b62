"""The trilinear interpolation with one lane per marker (what boxes of many
markers run) against eight lanes (what the small boxes of the oracle tests
run): the node velocities are added in the same order and every marker is
updated by the same operations, so a box has the same bits with either, for
every scheme, storage and forcing, populations pulled, read from the
node-moment field or from the node cache."""
import numpy as np
import pytest

import synth
from tests.gpu_helpers import require_cuda

pytestmark = pytest.mark.gpu

SCHEMES = [
    # kind, order, split, substeps
    ("fc", 2, "base", 1),
    ("fc", 2, "inside", 1),
    ("fc", 2, "inside", 3),
    ("fc", 2, "outside", 2),
    ("ebf", 2, "base", 1),
    ("mebf", 2, "base", 1),
    ("mebf", 2, "inside", 2),
    ("fc", 1, "base", 1),
    ("ibm", 2, "base", 1),
    ("ibm", 1, "base", 1),
]


# M = 41: a partial last group and warp
def _run(lanes, kind, order, split, n, storage, walls, kT, moments, M=41):
    from paper_1406_2211_gb300 import lbc
    nx, ny, nz = 16, 14, 12
    lat = lbc.lattice_desc(nx, ny, nz, collision="mrt", tau=0.9, body_force=(1e-5, 0, 0),
                           walls=walls, storage=storage)
    cpl = lbc.coupling_desc(kind, order, "trilinear", gamma=0.4 if M < 100 else 0.05, split=split, substeps=n)
    rng = np.random.default_rng(17)
    pos = rng.uniform(0.0, 1.0, (M, 3)) * [nx, ny, nz - 6.0] + [0.0, 0.0, 3.0]
    bonds = np.stack([np.arange(M - 1), np.arange(1, M)], axis=1)[::2]
    box = lbc.Box(lat, cpl, max_particles=M, max_bonds=len(bonds))
    if moments is not None:
        box.set_option(lbc.LBC_OPT_NODE_MOMENTS, moments)
    box.set_option(lbc.LBC_OPT_GATHER_LANES, lanes)
    if kT:
        box.set_thermal(kT, 5)
    box.set_populations(synth.random_populations((nz, ny, nx), seed=6, amp=1e-3))
    extra = {} if kind == "ibm" else dict(vel=0.15 * rng.standard_normal((M, 3)),
                                          mass=rng.uniform(5.0, 9.0, M),
                                          ext_force=1e-4 * rng.standard_normal((M, 3)))
    box.set_particles(pos, bonds=bonds, bond_k=0.0005, bond_r0=3.0, **extra)
    for steps in (1, 2, 3):
        box.step(steps)
    assert box.check() == 0
    out = [box.get_populations(), *box.get_particles(), *box.get_fields()]
    box.close()
    return out


def _same(lanes_args):
    a, b = _run(0, *lanes_args), _run(1, *lanes_args)
    for x, y in zip(a, b):
        assert np.isfinite(x).all()
        np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("kind,order,split,n", SCHEMES)
@pytest.mark.parametrize("storage", ["f64", "f32", "f16dev", "bf16dev"])
@pytest.mark.parametrize("walls", [False, True])
def test_one_lane_has_the_bits_of_eight(kind, order, split, n, storage, walls):
    require_cuda()
    _same((kind, order, split, n, storage, walls, 0.0, None))


@pytest.mark.parametrize("split,n", [("base", 1), ("inside", 2), ("outside", 2)])
@pytest.mark.parametrize("storage", ["f64", "f32"])
def test_one_lane_has_the_bits_of_eight_thermal(split, n, storage):
    require_cuda()
    _same(("fc", 2, split, n, storage, False, 1e-4, None))


@pytest.mark.parametrize("kind,split", [("fc", "base"), ("fc", "outside"), ("ibm", "base")])
@pytest.mark.parametrize("moments", [0, 1])
def test_one_lane_has_the_bits_of_eight_from_the_moments(kind, split, moments):
    require_cuda()
    _same((kind, 2, split, 1, "f32", False, 0.0, moments))


@pytest.mark.parametrize("storage,per_sm", [("f64", 32), ("f64", 56), ("f32", 96)])
@pytest.mark.parametrize("more", [0, 1])
@pytest.mark.parametrize("split,n", [("base", 1), ("inside", 2), ("outside", 1)])
def test_both_sides_of_the_lines(storage, per_sm, more, split, n):
    """Marker counts where the automatic choice passes from eight lanes to one."""
    require_cuda()
    import torch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    _same(("fc", 2, split, n, storage, False, 0.0, None, per_sm * sms + more))
