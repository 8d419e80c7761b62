"""Performance cases of the coupled lattice-Boltzmann step.

A case is one box (or one batch of boxes) as a simulation program sets it up,
and one pass is what such a program repeats: advance the box by a chunk of
time steps, then take the state.  The fluid comes back as the box's stored
populations, on the device: the caller owns the arena, the two population
arrays stand at its start, and after an even number of steps the state is in
the array that held it before.  The particles come back through
Box.get_particles, as a trajectory writer reads them, in the precision the
box computes in: FP64 for FP64 storage, FP32 for FP32 storage; in boxes of
16-bit storage the velocities and forces follow the stochastic rounding of
the fluid and are kept in 16 bits too (positions in FP32).

`exact` is the same scheme in plain torch FP64: populations streamed and
collided array by array, interpolation and spreading by indexing.
"""
import math

import numpy as np
import torch

from paper_1406_2211_gb300 import lbc

DEV = "cuda"
TDTYPE = {"f64": torch.float64, "f32": torch.float32, "f16dev": torch.float16,
          "bf16dev": torch.bfloat16}
ESIZE = {"f64": 8, "f32": 4, "f16dev": 2, "bf16dev": 2}

BASE = dict(family="box", nx=32, ny=32, nz=32, storage="f32", collision="bgk", tau=0.8,
            ghosts=False, walls=False, wall_u=0.0, body_g=0.0, kind="none", order=2,
            stencil="trilinear", split="base", substeps=1, gamma=1.0, particles="none",
            count=0, kT=0.0, stress=False, steps=20)


def make(name=None, **kw):
    c = dict(BASE)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    chains = dict(collision="mrt", kind="fc", gamma=5.0, split="inside", substeps=4,
                  particles="chains")
    return [
        # the smallest call in use: one force-coupled particle in a 32^3 FP64
        # box, the configuration the paper's coupling is checked on
        make("point_particle_32_f64", storage="f64", kind="fc", particles="points", count=1,
             steps=24),
        # one job of the serving ensemble on its own: launches and latency
        make("beads_64_f32", nx=64, ny=64, nz=64, kind="fc", gamma=4.0, particles="points",
             count=1000, steps=40),
        # one membrane shell between moving walls, reduced box of the shell
        # workload: a small IBM run
        make("shell_48_f32", nx=48, ny=48, nz=48, tau=1.0, walls=True, wall_u=0.05, kind="ibm",
             stencil="peskin4", particles="shells", count=1, steps=40),
        # the headline workload: bead chains in a 256^3 MRT fluid with the
        # multiple-time-step split
        make("bead_chains_256_f32", nx=256, ny=256, nz=256, tau=1.0, body_g=1e-6, count=2000,
             steps=16, **chains),
        # the same with 16-bit populations
        make("bead_chains_256_f16", nx=256, ny=256, nz=256, tau=1.0, body_g=1e-6, count=2000,
             storage="f16dev", steps=16, **chains),
        # chains in a thermal bath: fluctuating fluid and random forces
        make("thermal_chains_128_f32", nx=128, ny=128, nz=128, kT=1e-6, count=250, steps=20,
             **chains),
        # many membrane shells between moving walls (IBM, four-point stencil)
        make("shells_192_f32", nx=192, ny=192, nz=192, tau=1.0, walls=True, wall_u=0.05,
             kind="ibm", stencil="peskin4", particles="shells", count=64, steps=20),
        # a dense suspension of rigid spheres (modified EBF)
        make("spheres_128_f32", nx=128, ny=128, nz=128, tau=0.7, kind="mebf", stencil="peskin4",
             particles="spheres", count=500, steps=20),
        # plain fluid, every MRT rate set apart, ragged periodic box
        make("fluid_mrt_ragged_f32", nx=201, ny=161, nz=121, collision="mrt", ghosts=True,
             steps=40),
        # driven channel flow with 16-bit populations, rows of no special length
        make("channel_ragged_bf16", nx=150, ny=130, nz=110, storage="bf16dev", walls=True,
             body_g=1e-6, steps=40),
        # channel flow that writes its viscous stress as it goes
        make("channel_stress_f32", nx=192, ny=128, nz=96, walls=True, wall_u=0.02, body_g=1e-6,
             stress=True, steps=40),
        # the running batch of the serving loop: 16 boxes of edge 32-128 with
        # 1-5000 particles, FP32 and FP16 storage
        make("serving_16", family="batch", count=16, kind="fc", particles="points", steps=40),
    ]


def _odd_edge(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed kinds: sizes log-uniform over the range the
    kind is used in, every length (odd ones too), storages and options mixed."""
    kind = rng.choice(["points", "chains", "chains", "shells", "spheres", "fluid", "fluid", "batch"])
    storage = rng.choice(["f32", "f32", "f32", "f16dev", "bf16dev"])
    coll = rng.choice(["bgk", "mrt"])
    tau = round(rng.uniform(0.7, 1.2), 3)
    if kind == "points":
        e = [_odd_edge(rng, 32, 128) for _ in range(3)]
        small = e[0] * e[1] * e[2] <= 64 ** 3
        split = rng.choice(["base", "base", "outside"])
        order = rng.choice([1, 2, 2]) if split == "base" else 2
        return make(nx=e[0], ny=e[1], nz=e[2], storage=rng.choice([storage, "f64"]) if small else storage,
                    collision=coll, tau=tau, kind=rng.choice(["fc", "fc", "ebf", "mebf"]),
                    order=order, split=split, substeps=2 if split == "outside" else 1,
                    stencil=rng.choice(["trilinear", "trilinear", "peskin3", "peskin4"]),
                    gamma=round(rng.uniform(0.5, 1.0 if order == 1 else 4.0), 3), particles="points",
                    count=int(round(math.exp(rng.uniform(0.0, math.log(e[0] * e[1] * e[2] / 200.0))))),
                    steps=24 if small else 40)
    if kind == "chains":
        e = [_odd_edge(rng, 40, 240) for _ in range(3)]
        n = max(1, int(e[0] * e[1] * e[2] * rng.uniform(0.4, 1.0) * 2000 / 256 ** 3))
        return make(nx=e[0], ny=e[1], nz=e[2], storage=storage, collision=coll, tau=tau, kind="fc",
                    gamma=5.0, split="inside", substeps=4, particles="chains", count=n,
                    kT=rng.choice([0.0, 0.0, 1e-6]), steps=16)
    if kind == "shells":
        e = [_odd_edge(rng, 48, 180) for _ in range(3)]
        n = max(1, int(e[0] * e[1] * e[2] * rng.uniform(0.3, 1.0) * 64 / 192 ** 3))
        return make(nx=e[0], ny=e[1], nz=e[2], storage=storage, collision=coll, tau=tau, walls=True,
                    wall_u=0.05, kind="ibm", stencil=rng.choice(["peskin4", "peskin4", "peskin3"]),
                    particles="shells", count=n, steps=20)
    if kind == "spheres":
        e = [_odd_edge(rng, 32, 120) for _ in range(3)]
        n = max(1, int(e[0] * e[1] * e[2] * rng.uniform(0.3, 0.9) * 500 / 128 ** 3))
        return make(nx=e[0], ny=e[1], nz=e[2], storage="f32", collision=coll, tau=tau, kind="mebf",
                    stencil=rng.choice(["peskin4", "peskin4", "trilinear"]), particles="spheres",
                    count=n, steps=20)
    if kind == "fluid":
        e = [_odd_edge(rng, 40, 250) for _ in range(3)]
        walls = rng.random() < 0.5
        return make(nx=e[0], ny=e[1], nz=e[2], storage=storage, collision=coll, tau=tau,
                    ghosts=coll == "mrt" and rng.random() < 0.5, walls=walls,
                    wall_u=0.02 if walls else 0.0, body_g=1e-6 if walls else 0.0,
                    kT=rng.choice([0.0, 0.0, 1e-6]) if not walls else 0.0,
                    stress=walls and rng.random() < 0.4, steps=20)
    return make(family="batch", count=rng.randint(4, 16), kind="fc", particles="points",
                steps=40, tau=tau)


# ------------------------------------------------------------------ inputs
def _wave_fields(c, rng):
    """Density and velocity (torch FP64 on the device) of a few sound and
    shear waves of random direction and phase."""
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    ax = [torch.arange(n, dtype=torch.float64, device=DEV) for n in (nx, ny, nz)]
    out = torch.zeros((4, nz, ny, nx), dtype=torch.float64, device=DEV)
    for comp, amp in ((0, 2e-3), (1, 0.01), (2, 0.01), (3, 0.01)):
        for _ in range(2):
            k = rng.integers(-2, 3, 3)
            if not k.any():
                k[comp % 3] = 1
            px, py, pz = (2.0 * math.pi * int(k[a]) / n * ax[a] for a, n in enumerate((nx, ny, nz)))
            ph = float(rng.uniform(0.0, 2.0 * math.pi))
            out[comp] += amp * torch.sin(pz[:, None, None] + py[None, :, None] + px[None, None, :] + ph)
    return 1.0 + out[0], out[1:]


def _place(n, radius, box, walls, gap, rng):
    """n centres at least 2 radius + gap apart (periodic, or clear of the z
    walls), or as many as fit."""
    box = np.asarray(box, dtype=np.float64)
    lo, hi = np.zeros(3), box.copy()
    if walls:
        lo[2], hi[2] = radius + 2.5, box[2] - radius - 3.5
    got = np.zeros((0, 3))
    for _ in range(200):
        for p in lo + rng.uniform(0.0, 1.0, (256, 3)) * (hi - lo):
            d = p - got
            d[:, :2] -= box[:2] * np.rint(d[:, :2] / box[:2])
            if not walls:
                d[:, 2] -= box[2] * np.rint(d[:, 2] / box[2])
            if not len(got) or (d * d).sum(axis=1).min() >= (2 * radius + gap) ** 2:
                got = np.vstack([got, p])
                if len(got) == n:
                    return got
    return got


def _icosphere(levels):
    t = (1.0 + math.sqrt(5.0)) / 2.0
    v = [(0, s * 1, r * t) for s in (-1, 1) for r in (-1, 1)]
    v = np.array([np.roll(p, a) for a in range(3) for p in v], dtype=np.float64)
    d = np.linalg.norm(v[:, None] - v[None], axis=2)
    near = (d > 0.1) & (d < 2.1)
    faces = [(i, j, k) for i in range(12) for j in range(i) for k in range(j)
             if near[i, j] and near[j, k] and near[i, k]]
    v = [p / np.linalg.norm(p) for p in v]
    for _ in range(levels):
        mid, new = {}, []
        def m(a, b):
            key = (min(a, b), max(a, b))
            if key not in mid:
                mid[key] = len(v)
                p = v[a] + v[b]
                v.append(p / np.linalg.norm(p))
            return mid[key]
        for a, b, e in faces:
            ab, be, ea = m(a, b), m(b, e), m(e, a)
            new += [(a, ab, ea), (b, be, ab), (e, ea, be), (ab, be, ea)]
        faces = new
    edges = sorted({(min(p, q), max(p, q)) for a, b, e in faces for p, q in ((a, b), (b, e), (e, a))})
    return np.array(v), np.array(edges, dtype=np.int32)


_SHELL = []


def _particles(c, rng):
    """dict of set_particles arguments, or None."""
    box = (c["nx"], c["ny"], c["nz"])
    L = np.array(box, dtype=np.float64)
    kind, n = c["particles"], c["count"]
    if kind == "points":
        n = max(1, n)
        return dict(pos=rng.uniform(0.0, 1.0, (n, 3)) * L, vel=0.01 * rng.standard_normal((n, 3)),
                    mass=1.0)
    if kind == "chains":
        beads = 50
        head = rng.uniform(0.0, 1.0, (n, 1, 3)) * L
        step = rng.standard_normal((n, beads - 1, 3))
        step /= np.linalg.norm(step, axis=2, keepdims=True)
        pos = np.mod(np.cumsum(np.concatenate([head, step], axis=1), axis=1).reshape(-1, 3), L)
        idx = np.arange(n * beads, dtype=np.int32).reshape(n, beads)
        bonds = np.stack([idx[:, :-1].reshape(-1), idx[:, 1:].reshape(-1)], axis=1)
        return dict(pos=pos, vel=np.zeros_like(pos), mass=1.0, bonds=bonds, bond_k=10.0, bond_r0=1.0)
    if kind == "shells":
        if not _SHELL:
            _SHELL.extend(_icosphere(3))
        v, e = _SHELL
        R = 8.0
        centre = _place(n, R, box, True, 2.0, rng)
        pos = (centre[:, None, :] + R * v[None]).reshape(-1, 3)
        pos[:, :2] = np.mod(pos[:, :2], L[:2])
        bonds = (e[None] + len(v) * np.arange(len(centre), dtype=np.int32)[:, None, None]).reshape(-1, 2)
        r0 = np.tile(R * np.linalg.norm(v[e[:, 0]] - v[e[:, 1]], axis=1), len(centre))
        return dict(pos=pos, bonds=bonds, bond_k=0.05, bond_r0=r0)
    if kind == "spheres":
        R, m = 4.5, 400
        k = np.arange(m) + 0.5
        z = 1.0 - 2.0 * k / m
        th = math.pi * (3.0 - math.sqrt(5.0)) * k
        v = R * np.column_stack([np.sqrt(1.0 - z * z) * np.cos(th), np.sqrt(1.0 - z * z) * np.sin(th), z])
        centre = _place(n, R, box, False, 1.0, rng)
        pos = np.mod((centre[:, None, :] + v[None]).reshape(-1, 3), L)
        first = (np.arange(len(centre)) * m).astype(np.int32)
        ref = np.tile(v - v.mean(axis=0), (len(centre), 1))
        return dict(pos=pos, vel=0.002 * rng.standard_normal(pos.shape),
                    mass=4.0 / 3.0 * math.pi * R ** 3 / m,
                    rigid=dict(first=first, count=np.full(len(centre), m, dtype=np.int32), radius=R,
                               k=1.0, repulsion_k=0.1, ref=ref))
    return None


def _wall_velocity(c):
    return ((-c["wall_u"], 0.0, 0.0), (c["wall_u"], 0.0, 0.0))


def _rates(c):
    """MRT rates (shear, bulk, odd ghosts, even ghosts); 0 = the default."""
    return (1.0 / c["tau"], 1.1, 1.3, 1.6) if c["ghosts"] else (0.0, 0.0, 0.0, 0.0)


def _members(c, seed):
    """The boxes of a batch as cases of their own: edge log-uniform in
    32-128, 1-5000 particles, FP32 or FP16 storage."""
    if c["family"] != "batch":
        return [(c, seed)]
    rng = np.random.default_rng(20140609 + c["count"])      # the ensemble: the same for any inputs
    out = []
    for b in range(c["count"]):
        e = int(round(math.exp(rng.uniform(math.log(32), math.log(128)))))
        out.append((dict(c, family="box", nx=e, ny=e, nz=e, count=int(rng.integers(1, 5001)),
                         gamma=float(rng.uniform(0.5, 10.0)),
                         storage="f32" if rng.uniform() < 0.5 else "f16dev"), 1000 * seed + b))
    return out


def _box(c, seed):
    rng = np.random.default_rng(seed)
    lat = lbc.lattice_desc(c["nx"], c["ny"], c["nz"], collision=c["collision"], tau=c["tau"],
                           mrt_lambda=_rates(c), body_force=(c["body_g"], 0.0, 0.0),
                           walls=c["walls"], wall_velocity=_wall_velocity(c), storage=c["storage"])
    parts = _particles(c, rng)
    if parts is None:
        box = lbc.Box(lat)
    else:
        cpl = lbc.coupling_desc(c["kind"], c["order"], c["stencil"], gamma=c["gamma"],
                                split=c["split"], substeps=c["substeps"])
        box = lbc.Box(lat, cpl, max_particles=len(parts["pos"]),
                      max_bonds=len(parts["bonds"]) if "bonds" in parts else 0)
    rho, u = _wave_fields(c, rng)
    box.set_fields(rho.cpu().numpy(), u.cpu().numpy())
    if parts is not None:
        box.set_particles(**parts)
    if c["kT"] > 0.0:
        box.set_thermal(c["kT"], seed=int(seed) + 77)
    return box


def prepare(case, seed):
    boxes = []
    for c, s in _members(case, seed):
        box = _box(c, s)
        # set_fields leaves the state in the second population array, where
        # any even number of steps leaves it too; rows are padded to 32 bytes
        es = ESIZE[c["storage"]]
        nbytes = box.population_bytes()
        at = (nbytes + 255) // 256 * 256
        pitch = (c["nx"] * es + 31) // 32 * 32 // es
        pops = box.arena[at:at + nbytes].view(TDTYPE[c["storage"]])
        pops = pops.view(19, c["nz"], c["ny"], pitch)[..., :c["nx"]]
        boxes.append(dict(box=box, pops=pops, storage=c["storage"], kind=c["kind"]))
    state = dict(boxes=boxes, steps=case["steps"], sigma=None, batch=None)
    if case["stress"]:
        state["sigma"] = boxes[0]["box"].stress_output()
    if case["family"] == "batch":
        batch = lbc.Batch(len(boxes))
        for b in boxes:
            batch.add(b["box"], 1 << 40)         # long jobs: the batch keeps running
        state["batch"] = batch
    return state


def _particle_outputs(b):
    pos, vel, force = b["box"].get_particles()
    if b["storage"] == "f64":
        return [pos, vel, force]
    if b["storage"] == "f32":
        return [a.astype(np.float32) for a in (pos, vel, force)]
    return [pos.astype(np.float32)] + [torch.from_numpy(a).to(torch.bfloat16) for a in (vel, force)]


def run(state):
    if state["batch"] is not None:
        done = 0
        while done < state["steps"]:
            done += state["batch"].advance(state["steps"] - done)[0]
    else:
        state["boxes"][0]["box"].step(state["steps"])
    out = []
    for b in state["boxes"]:
        o = dict(pops=b["pops"])
        if b["kind"] == "ibm":                   # markers: positions only
            o["pos"] = _particle_outputs(b)[0]
        elif b["kind"] != "none":
            o["pos"], o["vel"], o["force"] = _particle_outputs(b)
        out.append(o)
    if state["sigma"] is not None:
        out[0]["sigma"] = state["sigma"]
    return out


def work(case):
    """Each time step reads and writes 19 populations per cell and the
    position and velocity of every particle; flops: the collision (about 230
    per cell) and interpolation and spreading (14 per stencil node each)."""
    total = dict(bytes=0.0, flops=0.0)
    for c, _ in _members(case, 0):
        cells = c["nx"] * c["ny"] * c["nz"]
        per = {"none": 0, "points": 1, "chains": 50, "shells": 642, "spheres": 400}[c["particles"]]
        m = per * c["count"]
        nodes = {"trilinear": 8, "peskin3": 27, "peskin4": 64}[c["stencil"]]
        couplings = {"ibm": 3}.get(c["kind"], 2 * c["substeps"] if c["split"] == "inside" else 2)
        total["bytes"] += c["steps"] * (cells * (38.0 * ESIZE[c["storage"]] + (24.0 if c["stress"] else 0.0)) +
                                        m * 96.0)
        total["flops"] += c["steps"] * (cells * 230.0 + m * nodes * 28.0 * couplings)
    return total


# ------------------------------------------------------------------ FP64 counterpart
_CI = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
       (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1),
       (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)]
_W = [1.0 / 3.0] + [1.0 / 18.0] * 6 + [1.0 / 36.0] * 12
_OPP = [0] + [i + 1 if i % 2 else i - 1 for i in range(1, 19)]


def _basis():
    """w-orthogonal moment basis: rows 1; c; c^2-1; five shear; six odd and
    three even ghost moments; and the relaxation group of each row."""
    rows = []
    for x, y, z in _CI:
        c2 = x * x + y * y + z * z
        rows.append([1, x, y, z, c2 - 1, 3 * x * x - c2, y * y - z * z, x * y, y * z, x * z,
                     (3 * c2 - 5) * x, (3 * c2 - 5) * y, (3 * c2 - 5) * z, (y * y - z * z) * x,
                     (z * z - x * x) * y, (x * x - y * y) * z, 3 * c2 * c2 - 6 * c2 + 1,
                     (2 * c2 - 3) * (3 * x * x - c2), (2 * c2 - 3) * (y * y - z * z)])
    return np.array(rows, dtype=np.float64).T, [0] * 4 + [1] + [2] * 5 + [3] * 6 + [4] * 3


def _philox(words, k0, k1):
    """Philox4x32-10 on int64 tensors holding 32-bit words."""
    mask = 0xFFFFFFFF

    def mul(a, b):
        lo, hi = a * (b & 0xFFFF), a * (b >> 16)
        return (hi + (lo >> 16)) >> 16, ((hi << 16) + lo) & mask
    x = list(words)
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
        h0, l0 = mul(0xD2511F53, x[0])
        h1, l1 = mul(0xCD9E8D57, x[2])
        x = [h1 ^ x[1] ^ k0, l1, h0 ^ x[3] ^ k1, l0]
    return x


def _normals(idx, step, stream, block, seed):
    full = lambda v: torch.full_like(idx, v)                                   # noqa: E731
    x = _philox([idx, full(step), full(stream), full(block)], seed & 0xFFFFFFFF, seed >> 32)
    u = [(w.double() + 0.5) * 2.0 ** -32 for w in x]
    out = []
    for a, b in ((0, 1), (2, 3)):
        r = torch.sqrt(-2.0 * torch.log(u[a]))
        out += [r * torch.cos(2.0 * math.pi * u[b]), r * torch.sin(2.0 * math.pi * u[b])]
    return out


class _Exact:
    def __init__(self, c, seed):
        self.c, self.step_no = c, 0
        rng = np.random.default_rng(seed)
        self.seed = int(seed) + 77
        parts = _particles(c, rng)
        rho, u = _wave_fields(c, rng)
        self.shape = (c["nz"], c["ny"], c["nx"])
        self.n3 = (c["nx"], c["ny"], c["nz"])
        self.g = torch.tensor([c["body_g"], 0.0, 0.0], dtype=torch.float64, device=DEV)
        E, group = _basis()
        w = np.array(_W)
        bk = (E * E) @ w
        lam_s, lam_b, lam_o, lam_e = _rates(c)
        lam_s = lam_s or 1.0 / c["tau"]
        lam_b = lam_b or lam_s
        lam = [0.0, lam_b, lam_s, lam_o or 1.0, lam_e or 1.0]
        mrt = c["collision"] == "mrt"
        gam = np.array([0.0 if q == 0 else 1.0 - (lam[q] if mrt else 1.0 / c["tau"]) for q in group])
        phi = np.array([0.0 if q == 0 else math.sqrt(3.0 * c["kT"] * b * (1.0 - g * g))
                        for q, b, g in zip(group, bk, gam)])
        t = lambda a: torch.as_tensor(a, dtype=torch.float64, device=DEV)     # noqa: E731
        self.E, self.back, self.gam, self.phi = t(E), t((E / bk[:, None]).T * w[:, None]), t(gam), t(phi)
        self.relax = t(((E / bk[:, None]).T * w[:, None]) @ (gam[:, None] * E))
        self.half = (0.5 * (1.0 + gam[4]), 0.5 * (1.0 + gam[5]))
        uw = _wall_velocity(c)
        self.bb = [[6.0 * _W[i] * sum(ci * v for ci, v in zip(_CI[i], uw[s])) for i in range(19)]
                   for s in range(2)]
        self.sigma = None
        # populations before streaming, as deviations from w_i
        fbar = self.feq(rho, u)
        self.f = torch.empty_like(fbar)
        for i, (x, y, z) in enumerate(_CI):
            self.f[i] = torch.roll(fbar[i], (-z, -y, -x), (0, 1, 2))
            if c["walls"] and z:
                at = -1 if z > 0 else 0
                self.f[i, at] = fbar[_OPP[i], at] - self.bb[1 if z > 0 else 0][_OPP[i]]
        self.Fa = torch.zeros((3,) + self.shape, dtype=torch.float64, device=DEV)
        self.parts = parts
        if parts is not None:
            self.r, m = t(parts["pos"]), len(parts["pos"])
            self.v = t(parts.get("vel", np.zeros((m, 3))))
            self.m = float(parts.get("mass", 1.0))
            self.Fh = torch.zeros_like(self.r)
            self.bonds = None
            if "bonds" in parts:
                b = torch.as_tensor(parts["bonds"].astype(np.int64), device=DEV)
                self.bonds = (b[:, 0], b[:, 1], parts["bond_k"],
                              t(np.broadcast_to(parts["bond_r0"], (len(b),)).copy()))
            self.rigid = parts.get("rigid")
            if self.rigid is not None:
                self.ref = t(self.rigid["ref"]).view(len(self.rigid["first"]), -1, 3)
        self.pull()

    def feq(self, rho, u):
        uu = 1.5 * (u * u).sum(0)
        out = torch.empty((19,) + self.shape, dtype=torch.float64, device=DEV)
        for i, (x, y, z) in enumerate(_CI):
            cu = x * u[0] + y * u[1] + z * u[2]
            out[i] = _W[i] * ((rho - 1.0) + rho * (3.0 * cu + 4.5 * cu * cu - uu))
        return out

    def pull(self):
        """fbar and its moments from the stored populations."""
        f = torch.empty_like(self.f)
        for i, (x, y, z) in enumerate(_CI):
            f[i] = torch.roll(self.f[i], (z, y, x), (0, 1, 2))
            if self.c["walls"] and z:
                at = 0 if z > 0 else -1
                f[i, at] = self.f[_OPP[i], at] + self.bb[0 if z > 0 else 1][i]
        self.fbar = f
        self.rd = f.sum(0)
        self.j = torch.stack([sum(ci[a] * f[i] for i, ci in enumerate(_CI) if ci[a]) for a in range(3)])

    def lb(self, half_force, g_weight=1.0):
        """One LB step; half_force: the force terms added to j for u1."""
        rho = 1.0 + self.rd
        u0 = self.j / rho
        u1 = u0 + (half_force + g_weight * self.g.view(3, 1, 1, 1)) / rho
        if self.c["stress"]:
            self.stress(rho, u0)
        neq = (self.fbar - self.feq(rho, u0)).view(19, -1)
        del self.fbar
        if self.c["kT"] > 0.0:
            post = self.gam[:, None] * (self.E @ neq)
            idx = torch.arange(neq.shape[1], dtype=torch.int64, device=DEV)
            sr = torch.sqrt(rho).view(-1)
            for blk in range(1, 5):
                for q, r in enumerate(_normals(idx, self.step_no, 0, blk, self.seed)):
                    if 4 * blk + q < 19:
                        post[4 * blk + q] += self.phi[4 * blk + q] * sr * r
            post = self.back @ post
        elif self.c["collision"] == "mrt":
            post = self.relax @ neq
        else:
            post = neq.mul_(1.0 - 1.0 / self.c["tau"])
        self.f = self.feq(rho, u1)
        self.f += post.view_as(self.f)
        self.pull()

    def stress(self, rho, u0):
        n = []
        for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (1, 2), (0, 2)):
            s = sum(ci[a] * ci[b] * self.fbar[i] for i, ci in enumerate(_CI) if ci[a] * ci[b])
            n.append(s - (self.rd / 3.0 if a == b else 0.0) - rho * u0[a] * u0[b])
        tr = (n[0] + n[1] + n[2]) / 3.0
        hb, hs = self.half
        self.sigma = torch.stack([hb * tr + hs * (x - tr) for x in n[:3]] + [hs * x for x in n[3:]])

    # ---- particles
    def wrap(self, r):
        r = r.clone()
        for a, n in enumerate(self.n3):
            if a < 2 or not self.c["walls"]:
                r[:, a] = torch.remainder(r[:, a], n)
        return r

    def image(self, d):
        d = d.clone()
        for a, n in enumerate(self.n3):
            if a < 2 or not self.c["walls"]:
                d[..., a] -= n * torch.round(d[..., a] / n)
        return d

    def stencil(self, r):
        """Flat node indices and weights, both (M, nodes)."""
        st = self.c["stencil"]
        idx, wt = [], []
        for a, n in enumerate(self.n3):
            X = r[:, a]
            if st == "trilinear":
                base, k = torch.floor(X), 2
            elif st == "peskin4":
                base, k = torch.floor(X) - 1, 4
            else:
                base, k = torch.floor(X + 0.5) - 1, 3
            node = base[:, None] + torch.arange(k, dtype=torch.float64, device=DEV)
            d = (X[:, None] - node).abs()
            if st == "trilinear":
                w = (1.0 - d).clamp(min=0.0)
            elif st == "peskin4":
                inner = (3 - 2 * d + torch.sqrt((1 + 4 * d - 4 * d * d).clamp(min=0.0))) / 8
                outer = (5 - 2 * d - torch.sqrt((-7 + 12 * d - 4 * d * d).clamp(min=0.0))) / 8
                w = torch.where(d <= 1.0, inner, outer)
            else:
                inner = (1 + torch.sqrt((1 - 3 * d * d).clamp(min=0.0))) / 3
                outer = (5 - 3 * d - torch.sqrt((-2 + 6 * d - 3 * d * d).clamp(min=0.0))) / 6
                w = torch.where(d <= 0.5, inner, outer)
            node = node.long()
            if a == 2 and self.c["walls"]:
                w = torch.where((node < 0) | (node >= n), torch.zeros_like(w), w)
                node = node.clamp(0, n - 1)
            else:
                node = torch.remainder(node, n)
            idx.append(node)
            wt.append(w)
        flat = (idx[2][:, :, None, None] * self.n3[1] + idx[1][:, None, :, None]) * self.n3[0] + \
            idx[0][:, None, None, :]
        w = wt[2][:, :, None, None] * wt[1][:, None, :, None] * wt[0][:, None, None, :]
        return flat.reshape(len(r), -1), w.reshape(len(r), -1)

    def velocity(self, sten, force=None, g=0.0):
        """Interpolated (j + force + g) / rho."""
        flat, w = sten
        inv = w / (1.0 + self.rd.view(-1)[flat])
        out = []
        for a in range(3):
            q = self.j[a].view(-1)[flat]
            if force is not None:
                q = q + force[a].reshape(-1)[flat]
            out.append(((q + g * self.g[a]) * inv).sum(1))
        return torch.stack(out, 1)

    def spread(self, sten, F):
        flat, w = sten
        out = torch.zeros((3, self.rd.numel()), dtype=torch.float64, device=DEV)
        for a in range(3):
            out[a].index_add_(0, flat.reshape(-1), (w * F[:, a:a + 1]).reshape(-1))
        return out.view((3,) + self.shape)

    def fint(self, r):
        F = torch.zeros_like(r)
        if self.bonds is not None:
            i, j, k, r0 = self.bonds
            d = self.image(r[j] - r[i])
            dist = d.norm(dim=1)
            f = d * (k * (dist - r0) / dist)[:, None]
            F.index_add_(0, i, f)
            F.index_add_(0, j, -f)
        if self.rigid is not None:
            nb, m = self.ref.shape[:2]
            y = r.view(nb, m, 3)
            y = y[:, :1] + self.image(y - y[:, :1])
            X = y.mean(1, keepdim=True)
            A = (y - X).transpose(1, 2) @ self.ref
            U, _, Vh = torch.linalg.svd(A)
            R = U @ Vh
            f = -self.rigid["k"] * (y - X - self.ref @ R.transpose(1, 2))
            d = self.image(X[:, 0][None] - X[:, 0][:, None])
            dist = d.norm(dim=2) + 1e9 * torch.eye(nb, dtype=torch.float64, device=DEV)
            gap = dist - 2.0 * self.rigid["radius"]
            mag = torch.where(gap < 1.0, self.rigid["repulsion_k"] * (1.0 - gap) / dist, torch.zeros_like(gap))
            rep = -(mag[..., None] * d).sum(1)
            F += (f + rep[:, None] / m).reshape(-1, 3)
        return F

    def couple(self, v, u, Fi, s, sub):
        c = self.c
        if c["kind"] == "mebf":
            return -(v - u) / (s * (1.0 / self.m + 1.0)) - Fi / (1.0 + self.m)
        gam = 1.0 if c["kind"] == "ebf" else c["gamma"]
        zeta = 0.0
        if c["kT"] > 0.0:
            idx = torch.arange(len(v), dtype=torch.int64, device=DEV)
            r = _normals(idx, self.step_no, 8 + sub, 0, self.seed)
            zeta = math.sqrt(2.0 * c["kT"] * gam / s) * torch.stack(r[:3], 1)
        if c["order"] == 1:
            return -gam * (v - u) + zeta
        al, be = gam * s / self.m, gam * s
        return -(gam * (v - u) + 0.5 * al * Fi - zeta) / (1.0 + 0.5 * al + 0.5 * be)

    def inside_half(self, before):
        n = self.c["substeps"]
        dt = 0.5 / n
        acc = torch.zeros_like(self.Fa)
        for k in range(n):
            self.r = self.wrap(self.r + 0.5 * dt * self.v)
            Fi, st = self.fint(self.r), self.stencil(self.r)
            force = 0.5 * (self.Fa + acc) if before else 0.5 * acc
            u = self.velocity(st, force, (0.5 if before else 0.0) + 0.5 * k / n)
            self.Fh = self.couple(self.v, u, Fi, dt, (0 if before else n) + k)
            self.v = self.v + dt / self.m * (self.Fh + Fi)
            acc += self.spread(st, -self.Fh) / n
            self.r = self.wrap(self.r + 0.5 * dt * self.v)
        return acc

    def outside_verlet(self):
        n = self.c["substeps"]
        dt = 0.5 / n
        for _ in range(n):
            self.r = self.wrap(self.r + 0.5 * dt * self.v)
            self.v = self.v + dt / self.m * self.fint(self.r)
            self.r = self.wrap(self.r + 0.5 * dt * self.v)

    def step(self):
        c = self.c
        if self.parts is None:
            self.lb(0.0)
        elif c["kind"] == "ibm":
            Xt = self.wrap(self.r + 0.5 * self.velocity(self.stencil(self.r), 0.5 * self.Fa, 0.5))
            self.Fh, st = self.fint(Xt), self.stencil(Xt)
            self.r = self.wrap(self.r + 0.5 * self.velocity(st, 0.5 * self.Fa, 0.5))
            Fb = self.spread(st, self.Fh)
            self.lb(0.5 * (self.Fa + Fb))
            self.Fa = Fb
            self.r = self.wrap(self.r + 0.5 * self.velocity(st, 0.5 * Fb, 0.5))
        elif c["order"] == 1:
            Fi, st = self.fint(self.r), self.stencil(self.r)
            self.Fh = self.couple(self.v, self.velocity(st), Fi, 1.0, 0)
            self.v = self.v + (self.Fh + Fi) / self.m
            self.lb(self.spread(st, -self.Fh))
            self.r = self.wrap(self.r + self.v)
        elif c["split"] == "inside":
            Fb = self.inside_half(True)
            self.lb(0.5 * (self.Fa + Fb))
            self.Fa = self.inside_half(False)
        elif c["split"] == "outside":
            zero = torch.zeros_like(self.v)
            st = self.stencil(self.r)
            Fh = self.couple(self.v, self.velocity(st, 0.5 * self.Fa, 0.5), zero, 0.5, 0)
            self.v = self.v + 0.5 / self.m * Fh
            Fb = self.spread(st, -Fh)
            self.outside_verlet()
            self.lb(0.5 * (self.Fa + Fb))
            self.outside_verlet()
            st = self.stencil(self.r)
            self.Fh = self.couple(self.v, self.velocity(st), zero, 0.5, 1)
            self.Fa = self.spread(st, -self.Fh)
            self.v = self.v + 0.5 / self.m * self.Fh
        else:
            self.r = self.wrap(self.r + 0.5 * self.v)
            Fi, st = self.fint(self.r), self.stencil(self.r)
            Fh = self.couple(self.v, self.velocity(st, 0.5 * self.Fa, 0.5), Fi, 0.5, 0)
            self.v = self.v + 0.5 / self.m * (Fh + Fi)
            self.lb(0.5 * (self.Fa + self.spread(st, -Fh)))
            self.Fh = self.couple(self.v, self.velocity(st), Fi, 0.5, 1)
            self.Fa = self.spread(st, -self.Fh)
            self.v = self.v + 0.5 / self.m * (self.Fh + Fi)
            self.r = self.wrap(self.r + 0.5 * self.v)
        self.step_no += 1


def exact(case, seed):
    out = []
    for c, s in _members(case, seed):
        sim = _Exact(c, s)
        for _ in range(c["steps"]):
            sim.step()
        f = sim.f
        if ESIZE[c["storage"]] == 2:             # stored divided by w_i
            f = f / torch.tensor(_W, dtype=torch.float64, device=DEV).view(19, 1, 1, 1)
        o = dict(pops=f)
        if sim.parts is not None:
            o["pos"] = sim.r
            if c["kind"] != "ibm":
                o["vel"], o["force"] = sim.v, sim.Fh
        if c["stress"]:
            o["sigma"] = sim.sigma
        out.append(o)
        del sim
    return out
