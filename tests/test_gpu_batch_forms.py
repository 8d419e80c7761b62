"""A member's bits must not depend on how its particle work is launched:
the box on its own, in a batch with one launch per operation and in a batch
with a stream of its own, for 16-bit and FP32 storage, with and without walls
(16-bit populations are products, and each kernel is compiled for itself), in
a box dense with markers so that a difference in the last place of one
node's density shows."""
import numpy as np
import pytest

import synth
from tests.gpu_helpers import require_cuda

pytestmark = pytest.mark.gpu

M = 7601
SCHEMES = {"fc": ("fc", "base", 1), "fc_inside": ("fc", "inside", 2), "ibm": ("ibm", "base", 1)}


def make_member(scheme, storage, walls, stencil="trilinear", moments=None, seed=40, count=M,
                reach=3.0):
    """reach: how near the markers start to the walls."""
    from paper_1406_2211_gb300 import lbc
    kind, split, n = SCHEMES[scheme]
    nx, ny, nz = 26, 24, 22
    lat = lbc.lattice_desc(nx, ny, nz, tau=0.8, walls=walls, storage=storage,
                           wall_velocity=((0.01, 0, 0), (-0.01, 0, 0)) if walls else ((0,) * 3,) * 2)
    cpl = lbc.coupling_desc(kind, 2, stencil, gamma=0.05, split=split, substeps=n)
    box = lbc.Box(lat, cpl, max_particles=count)
    if moments is not None and n == 1:
        box.set_option(lbc.LBC_OPT_NODE_MOMENTS, moments)
    box.set_option(lbc.LBC_OPT_LB_PAIR, 0)      # the batched LB kernels take one cell per thread
    box.set_populations(synth.random_populations((nz, ny, nx), seed=seed, amp=1e-3))
    rng = np.random.default_rng(seed)
    pos = rng.uniform(0.0, 1.0, (count, 3)) * [nx, ny, nz - 2.0 * reach] + [0.0, 0.0, reach]
    extra = {} if kind == "ibm" else dict(vel=0.1 * rng.standard_normal((count, 3)), mass=3.0)
    box.set_particles(pos, **extra)
    return box


def state(box):
    return [box.get_populations(), *box.get_particles()]


def advance(boxes, launch, steps=5):
    from paper_1406_2211_gb300 import lbc
    batch = lbc.Batch(len(boxes))
    batch.set_launch(launch)
    for b in boxes:
        assert batch.add(b, steps)
    while len(batch):
        batch.advance(steps)
    batch.close()
    return [state(b) for b in boxes]


def assert_same(a, b):
    for x, y in zip(a, b):
        assert np.isfinite(x).all()
        np.testing.assert_array_equal(x, y)


@pytest.mark.parametrize("scheme", list(SCHEMES))
@pytest.mark.parametrize("storage", ["f16dev", "bf16dev", "f32"])
@pytest.mark.parametrize("walls,reach", [(False, 0.0), (True, 3.0), (True, 1.0)])
@pytest.mark.parametrize("moments", [0, 1])
def test_box_and_batch_forms_give_the_same_bits(scheme, storage, walls, reach, moments):
    require_cuda()
    args = (scheme, storage, walls)
    kw = dict(moments=moments, reach=reach)
    box = make_member(*args, **kw)
    box.step(5)
    assert box.check() == 0
    alone = state(box)
    for launch in ("batched", "streams"):
        assert_same(advance([make_member(*args, **kw)], launch)[0], alone)


@pytest.mark.parametrize("stencil", ["peskin4", "peskin3"])
@pytest.mark.parametrize("storage", ["f16dev", "bf16dev", "f32"])
@pytest.mark.parametrize("walls", [False, True])
def test_wide_stencils_of_box_and_batch_forms(stencil, storage, walls):
    require_cuda()
    kw = dict(stencil=stencil, count=1501)
    box = make_member("fc", storage, walls, **kw)
    box.step(5)
    alone = state(box)
    for launch in ("batched", "streams"):
        assert_same(advance([make_member("fc", storage, walls, **kw)], launch)[0], alone)
