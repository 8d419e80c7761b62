"""The base split's opening drift, a launch of its own or part of the
interpolation by the number of markers: a box on either side of each line
against the FP64 oracle, with fields set between steps (which must keep a
requested re-sort) and markers fast enough to leave their bins, then the same
box with fewer and with more markers (the choice is made again).  Bounds as in
test_gpu_coupling (FP64 storage: roundoff)."""
import numpy as np
import pytest

from oracle import coupling as OC
from oracle import lattice as OLat
from oracle import lb as OL
from oracle import sim as OS
from tests.gpu_helpers import require_cuda

pytestmark = pytest.mark.gpu

FEW, MANY = 4096, 96 * 152


def _particles(M, shape, seed):
    nz, ny, nx = shape
    rng = np.random.default_rng(seed)
    pos = rng.uniform(0.0, 1.0, (M, 3)) * [nx, ny, nz]
    vel = 0.3 * rng.choice([-1.0, 1.0], (M, 3)) * rng.uniform(0.5, 1.0, (M, 3))
    bonds = np.stack([np.arange(0, M - 1, 2), np.arange(1, M, 2)[: len(range(0, M - 1, 2))]], axis=1)
    return dict(pos=pos, vel=vel, mass=np.full(M, 4.0), bonds=bonds, bond_k=0.001, bond_r0=2.0)


@pytest.mark.parametrize("counts", [(FEW, FEW + 1, FEW), (MANY, MANY + 1, 37)])
def test_either_side_of_the_lines_matches_oracle(counts):
    require_cuda()
    from paper_1406_2211_gb300 import lbc
    shape = (26, 28, 30)
    nz, ny, nx = shape
    M = max(counts)
    lat = lbc.lattice_desc(nx, ny, nz, tau=0.9, storage="f64")
    cpl = lbc.coupling_desc("fc", 2, "trilinear", gamma=0.05)
    box = lbc.Box(lat, cpl, max_particles=M, max_bonds=M)
    rho, u = np.ones(shape), np.zeros((3,) + shape)
    u[0] = 0.03
    feq = OLat.equilibrium(rho, u)
    for seed, count in enumerate(counts):
        parts = _particles(count, shape, seed)
        box.set_fields(rho, u)
        box.set_particles(**parts)
        op = dict(parts, pos=OC.wrap_positions(parts["pos"], shape, False))
        sm = OS.Sim(shape, OL.LBParams(collision="bgk", tau=0.9),
                    OS.CouplingParams("fc", 2, "trilinear", gamma=0.05), OC.Particles(**op),
                    fbar=feq.copy())
        for nsteps in (1, 4, 2):
            box.step(nsteps)
            for _ in range(nsteps):
                sm.step()
            box.set_fields(rho, u)
            sm.fbar = feq.copy()
            sm.Fa = np.zeros_like(u)
        pos, vel, fh = box.get_particles()
        assert np.abs(OC.min_image(pos - sm.parts.pos, shape, False)).max() < 1e-11
        assert np.abs(vel - sm.parts.vel).max() < 1e-11
        assert np.abs(fh - sm.last_Fh).max() < 1e-11
        assert box.check() == 0
    box.close()
