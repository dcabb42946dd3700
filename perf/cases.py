"""Benchmark cases: what users of the library run, through its Python binding.

A case is a dict of plain numbers and texts.  Three kinds of work:

``lattice``   one lattice: `steps` coupled steps (``lbmd_step``), then the whole updated state read
              back into device tensors (``lbmd_get_populations_dev``, ``lbmd_get_particles_dev``).
``observe``   looking at a state between steps: the FP64 totals (``lbmd_diagnostics``) and the
              fields (``lbmd_get_fields_dev``).
``replicas``  serving: many independent lattices advanced together, `chunk` steps per
              ``lbmd_batch_step`` + ``lbmd_batch_poll`` as the serving loop does, then the
              densities and particles of every replica read back to the host.

Three systems, all from seeded generators: ``noise`` (a mixture demixing from +-1 % noise),
``droplets`` (an A-rich slab and droplets at bulk coexistence, particles with solvation coupling)
and ``chains`` (charged bead-spring chains in a demixing mixture).

`exact` restates the model in 64 bits with plain torch operations.
"""
import math

import numpy as np
import torch

from paper_1306_0788_gb300 import inputs, serving
from paper_1306_0788_gb300 import lbmd as L

DENSITY = 78.4  # mean density per component of the droplet and chain systems
STORAGES = {"fp32": L.LBMD_STORAGE_FP32, "fp16": L.LBMD_STORAGE_FP16_SHIFTED, "bf16": L.LBMD_STORAGE_BF16_SHIFTED}
CHAIN = 50  # beads per chain
SPACING = 2.5  # edge of the cells that hold at most one particle each


def _lattice(name, dims, system, particles, steps, storage="fp32", collision="bgk", substeps=1):
    return dict(name=name, kind="lattice", nx=dims[0], ny=dims[1], nz=dims[2], system=system, particles=particles,
                steps=steps, storage=storage, collision=collision, substeps=substeps)


def listed():
    return [
        # the smallest single system: 32^3 from noise with 64 friction-coupled particles
        _lattice("noise_32", (32, 32, 32), "noise", 64, 50),
        # a small box of no round size, fluid only: a short parameter study
        _lattice("fluid_45x37x29", (45, 37, 29), "noise", 0, 50),
        # a desktop-size system that stays in the GPU's L2
        _lattice("droplets_64", (64, 64, 64), "droplets", 1000, 50),
        # polyelectrolyte chains with ten particle updates per lattice step
        _lattice("chains_80_substeps", (80, 80, 80), "chains", 800, 10, substeps=10),
        # thermal fluctuations (MRT with noise) in a box of no round size
        _lattice("thermal_100x90x110", (100, 90, 110), "droplets", 1000, 20, collision="mrt"),
        # the middle of the range, at the particle density of the 256^3 system
        _lattice("droplets_128", (128, 128, 128), "droplets", 2500, 20),
        # the interface-adsorption system: 256^3, 2e4 particles, in FP32 ...
        _lattice("droplets_256", (256, 256, 256), "droplets", 20000, 10),
        # ... with populations stored in 16 bits ...
        _lattice("droplets_256_fp16", (256, 256, 256), "droplets", 20000, 10, storage="fp16"),
        # ... and with thermal fluctuations
        _lattice("thermal_256", (256, 256, 256), "droplets", 20000, 10, collision="mrt"),
        # the largest system: 512^3 demixing with 1000 chains of 50 charged beads
        _lattice("chains_512", (512, 512, 512), "chains", 50000, 10),
        # monitoring: totals and fields of a 256^3 state
        dict(name="observe_256", kind="observe", nx=256, ny=256, nz=256, particles=20000, storage="fp32"),
        # serving: 24 replicas of the request distribution (edges 16 to 128, up to 5000 particles)
        dict(name="replicas_24", kind="replicas", chunk=25, steps=250,
             edges="18 22 27 31 36 40 45 50 54 59 63 68 73 77 82 86 91 96 100 105 109 114 119 125",
             particles="30 0 600 300 1200 0 2500 700 3900 1800 0 5000 900 3100 2200 4500 100 0 3600 1500 2800 5000 0 4100"),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choices(("lattice", "observe", "replicas"), (8, 1, 1))[0]
    if kind == "replicas":
        n = rng.randint(4, 24)
        edges = [rng.randint(16, 128) for _ in range(n)]
        cap = [int(0.5 * int(e // SPACING) ** 3) for e in edges]
        return dict(kind=kind, chunk=25, steps=rng.choice((100, 150, 200)), edges=" ".join(map(str, edges)),
                    particles=" ".join(str(min(rng.randint(0, 5000), c)) for c in cap))
    edge = _log_uniform(rng, 24, 300)
    dims = [max(20, round(edge * rng.uniform(0.8, 1.25))) for _ in range(3)]
    if rng.random() < 0.3:
        dims = [max(32, 32 * round(d / 32)) for d in dims]
    nx, ny, nz = dims
    most = int(0.25 * math.prod(int(d // SPACING) for d in dims))
    particles = min(most, round(_log_uniform(rng, 50, 20000))) if rng.random() < 0.8 else 0
    storage = rng.choices(("fp32", "fp16", "bf16"), (6, 2, 1))[0]
    if kind == "observe":
        return dict(kind=kind, nx=nx, ny=ny, nz=nz, particles=particles, storage=storage)
    system = rng.choices(("noise", "droplets", "chains"), (2, 5, 2))[0]
    substeps = 1
    if system == "chains":
        dims = nx, ny, nz = [max(40, d) for d in dims]
        particles = CHAIN * max(2, min(_chain_places(dims) // 4, particles // CHAIN))
        substeps = rng.choice((1, 1, 5, 10))
    sites = nx * ny * nz
    steps = 50 if sites < 300_000 else 20 if sites < 3_000_000 else 10
    case = _lattice("", (nx, ny, nz), system, particles, steps, storage,
                    "mrt" if substeps == 1 and rng.random() < 0.25 else "bgk", substeps)
    del case["name"]
    return case


# ------------------------------------------------------------------ inputs

def _dims(case):
    return case["nx"], case["ny"], case["nz"]


def _model(case):
    """Couplings, thermal energy and particle type of a system; energies of the chains in units of kT."""
    system = case.get("system", "droplets")
    m = dict(g=0.0214, kT=0.01, kappa=(-0.001, -0.002), lam=(0.0, 0.0), gamma=1.0, mass=200.0, wca=(1.0, 1.0),
             dh=None, fene=None)
    if system == "noise":
        m.update(g=1.4, kT=1e-4, kappa=(0.0, 0.0))
    elif system == "chains":
        kT = 0.01
        m.update(g=1.4 / DENSITY, kT=kT, kappa=(-5e-4 * kT, 5e-4 * kT), lam=(0.01 * kT, 0.0), mass=100.0, wca=(kT, 1.0),
                 dh=(kT, 0.25, 3.0), fene=(30.0 * kT, 1.5))
    return m


def _densities(case, seed):
    """rho_A, rho_B [nz, ny, nx] as FP32 host arrays (made on the GPU)."""
    nx, ny, nz = _dims(case)
    gen = torch.Generator("cuda").manual_seed(seed)
    noise = torch.rand((2, nz, ny, nx), generator=gen, device="cuda").mul_(0.02).sub_(0.01)
    system = case.get("system", "droplets")
    if system != "droplets":
        scale = 1.0 if system == "noise" else DENSITY
        rho = noise.add_(1.0).mul_(scale)
        return rho[0].cpu().numpy(), rho[1].cpu().numpy()
    z = torch.arange(nz, device="cuda", dtype=torch.float32)[:, None, None]
    y = torch.arange(ny, device="cuda", dtype=torch.float32)[None, :, None]
    x = torch.arange(nx, device="cuda", dtype=torch.float32)[None, None, :]
    width = 4.0 if min(nx, ny, nz) >= 64 else 2.0
    phi = (0.5 * (1.0 + torch.tanh(torch.minimum(z - nz / 4, 3 * nz / 4 - z) / width))).expand(nz, ny, nx).clone()
    g = np.random.default_rng(seed)
    for _ in range(8):  # droplets in the B-rich quarter around z = 0, where they fit
        r = g.uniform(1 / 32, 1 / 10) * min(nx, ny, nz)
        c = (g.uniform(0, nx), g.uniform(0, ny), g.uniform(-0.05, 0.05) * nz)
        d2 = 0.0
        for a, ca, n in ((x, c[0], nx), (y, c[1], ny), (z, c[2], nz)):
            d = a - ca
            d2 = d2 + (d - n * torch.round(d / n)) ** 2
        phi = torch.maximum(phi, 0.5 * (1.0 + torch.tanh((r - torch.sqrt(d2)) / width)))
    hi, lo = 1.9103 * DENSITY, 0.0897 * DENSITY  # bulk coexistence at g rho = 1.68
    rA = (lo + (hi - lo) * phi) * (1.0 + noise[0])
    rB = (hi - (hi - lo) * phi) * (1.0 + noise[1])
    return rA.cpu().numpy(), rB.cpu().numpy()


def _flow(case, seed):
    """A shear flow of amplitude 0.05 in each direction, u [nz, ny, nx, 3] FP32."""
    nx, ny, nz = _dims(case)
    a = np.random.default_rng(seed + 3).uniform(0, 2 * np.pi, size=3)
    wave = lambda n, k: 0.05 * np.sin(2 * np.pi * np.arange(n) / n + a[k])  # noqa: E731
    u = np.empty((nz, ny, nx, 3), dtype=np.float32)
    u[..., 0] = wave(ny, 0)[None, :, None]
    u[..., 1] = wave(nz, 1)[:, None, None]
    u[..., 2] = wave(nx, 2)[None, None, :]
    return u


def _chain_places(dims):
    return (dims[0] // 32) * (dims[1] // 4) * (dims[2] // 4)


def _chains(n, dims, seed):
    """Helical coils of CHAIN beads, bond length 0.97, each in a tube of its own (at least 1.6 apart):
    positions, bonds, charges +1 and -1 by chain."""
    g = np.random.default_rng(seed)
    m = n // CHAIN
    places = g.choice(_chain_places(dims), size=m, replace=False)
    ty, tz = dims[1] // 4, dims[2] // 4
    origin = np.stack([places // (ty * tz) * 32.0, places // tz % ty * 4.0 + 2.0, places % tz * 4.0 + 2.0], axis=1)
    k = np.arange(CHAIN)
    turn = 2 * math.asin(math.sqrt(0.97 ** 2 - 0.6 ** 2) / 2.4)
    angle = g.uniform(0, 2 * np.pi, size=m)[:, None] + turn * k * np.where(g.random(m) < 0.5, 1.0, -1.0)[:, None]
    x = np.stack([origin[:, :1] + 0.6 * k, origin[:, 1:2] + 1.2 * np.cos(angle), origin[:, 2:] + 1.2 * np.sin(angle)],
                 axis=2).reshape(-1, 3) + g.uniform(-0.02, 0.02, size=(n, 3))
    first = (np.arange(m)[:, None] * CHAIN + k[:-1]).ravel()
    q = np.where(np.arange(n) // CHAIN % 2 == 0, 1.0, -1.0)
    return x % np.array(dims, dtype=np.float64), np.stack([first, first + 1], axis=1).astype(np.int32), q


def _particles(case, seed):
    """Positions, velocities, bonds and charges (None where the system has none)."""
    n, dims, m = case["particles"], _dims(case), _model(case)
    if n == 0:
        return None
    v = np.random.default_rng(seed + 2).normal(scale=math.sqrt(m["kT"] / m["mass"]), size=(n, 3))
    if case.get("system") == "chains":
        x, bonds, q = _chains(n, dims, seed + 1)
        return x, v, bonds, q
    return inputs.spaced_particles(n, dims, SPACING, seed=seed + 1), v, None, None


def _requests(case, seed):
    g = np.random.default_rng(seed)
    return [dict(edge=int(e), np=int(n), g=float(g.uniform(1.2, 2.1)), gamma=float(g.uniform(0.1, 2.0)),
                 seed=int(g.integers(0, 2 ** 31 - 1)), steps=10 ** 9)
            for e, n in zip(case["edges"].split(), case["particles"].split())]


# ------------------------------------------------------------------ states

class Context:
    """One lattice as a user's program holds it, and the tensors its results go to."""

    def __init__(self, case, seed):
        dims, m = _dims(case), _model(case)
        rA, rB = _densities(case, seed)
        self.case = case
        rho0 = (float(rA.mean()), float(rB.mean()))
        mrt = case.get("collision") == "mrt"
        self.ctx, _ = L.lbmd_create(L.params(
            dims, tau_r=1.0, g_AB=m["g"], kT=m["kT"], seed=seed, storage=STORAGES[case["storage"]], rho0=rho0,
            collision=L.LBMD_COLLISION_MRT if mrt else L.LBMD_COLLISION_BGK, md_substeps=case.get("substeps", 1)))
        shape = dims[::-1]
        L.lbmd_init_fluid(self.ctx, rA, rB, _flow(case, seed) if case["kind"] == "observe" else None)
        if case["kind"] == "observe":
            self.rho = [torch.empty(shape, dtype=torch.float32, device="cuda") for _ in range(2)]
            self.u = torch.empty(shape + (3,), dtype=torch.float32, device="cuda")
        else:
            self.f = [torch.empty((19,) + shape, dtype=torch.float32, device="cuda") for _ in range(2)]
        parts = _particles(case, seed)
        self.xvf = None
        if parts is not None:
            x, v, bonds, q = parts
            L.lbmd_set_types(self.ctx, [L.lbmd_ptype(*m["kappa"], *m["lam"], m["gamma"], m["mass"])],
                             [L.lbmd_pair(0, 0, *m["wca"])])
            if m["dh"]:
                L.lbmd_set_debye_hueckel(self.ctx, *m["dh"])
            L.lbmd_set_particles(self.ctx, x, v, np.zeros(len(x), dtype=np.int32), q)
            if bonds is not None:
                L.lbmd_set_bonds(self.ctx, bonds, L.LBMD_BOND_FENE, *m["fene"])
            self.xvf = torch.empty((3, len(x), 3), dtype=torch.float64, device="cuda")

    def __del__(self):
        if getattr(self, "ctx", None) is not None:
            L.lbmd_destroy(self.ctx)
            self.ctx = None


class Replicas:
    def __init__(self, case, seed):
        self.case = case
        self.requests = _requests(case, seed)
        self.server = serving.Server(max_slots=64, chunk=case["chunk"])
        self.slots = [serving.admit(self.server.batch, r) for r in self.requests]

    def __del__(self):
        if getattr(self, "server", None) is not None:
            self.server.close()
            self.server = None


def prepare(case, seed):
    return Replicas(case, seed) if case["kind"] == "replicas" else Context(case, seed)


def run(state):
    case = state.case
    if case["kind"] == "replicas":
        b = state.server.batch
        for _ in range(case["steps"] // case["chunk"]):
            L.lbmd_batch_step(b, case["chunk"])
            L.lbmd_batch_poll(b, state.server.max_slots)
        out = []
        for slot, r in zip(state.slots, state.requests):
            rA, rB, _ = L.lbmd_batch_get_fields(b, slot, (r["edge"],) * 3, want_u=False)
            # FP64 arrays that hold what the library keeps in FP32
            out.append([rA, rB] + [a.astype(np.float32) for a in L.lbmd_batch_get_particles(b, slot, r["np"])])
        # one array per quantity, the replicas one after another
        return {name: np.concatenate([o[k].ravel() for o in out])
                for k, name in enumerate(("rho_A", "rho_B", "x", "v", "force"))}
    ctx = state.ctx
    if case["kind"] == "observe":
        totals = L.lbmd_diagnostics(ctx)
        L.lbmd_get_fields_dev(ctx, state.rho[0].data_ptr(), state.rho[1].data_ptr(), state.u.data_ptr())
        return {"totals": totals, "rho_A": state.rho[0], "rho_B": state.rho[1], "u": state.u}
    L.lbmd_step(ctx, case["steps"])
    for comp in (0, 1):
        L.lbmd_get_populations_dev(ctx, comp, state.f[comp].data_ptr())
    out = {"f_A": state.f[0], "f_B": state.f[1]}
    if state.xvf is not None:
        L.lbmd_get_particles_dev(ctx, *(t.data_ptr() for t in state.xvf))
        out.update(zip(("x", "v", "force"), state.xvf.float()))  # the library keeps them in FP32
    return out


def work(case):
    """Each population read once and written once per step (FP32: 38 x 4 B each way; 16 bits: 36 x 2 B
    and the two FP32 rest populations), the particle state likewise; the results written once."""
    if case["kind"] == "replicas":
        sites = sum(int(e) ** 3 for e in case["edges"].split())
        particles = sum(map(int, case["particles"].split()))
        return {"bytes": case["steps"] * (304 * sites + 104 * particles) + 8 * sites + 36 * particles,
                "flops": case["steps"] * (500 * sites + 3000 * particles)}
    sites, particles = math.prod(_dims(case)), case["particles"]
    state = 152 if case["storage"] == "fp32" else 80
    if case["kind"] == "observe":
        return {"bytes": (state + 20) * sites + 16 * particles, "flops": 250 * sites + 6 * particles}
    per_site = 1700 if case["collision"] == "mrt" else 500
    return {"bytes": case["steps"] * (2 * state * sites + 104 * particles * case["substeps"])
            + (state + 152) * sites + 36 * particles,
            "flops": case["steps"] * (per_site * sites + 3000 * particles * case["substeps"])}


# ------------------------------------------------------------------ the model in 64 bits

C = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
              (1, 1, 0), (-1, -1, 0), (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1),
              (0, 1, 1), (0, -1, -1), (0, 1, -1), (0, -1, 1)])
W = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)


def _philox(counter, seed):
    """Philox4x32-10 of four int64 tensors that hold 32-bit words, under the 64-bit key `seed`."""
    low = 0xFFFFFFFF
    c0, c1, c2, c3 = counter
    k0, k1 = seed & low, seed >> 32 & low
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57  # the low 64 bits, also where the sign is lost
        c0, c1, c2, c3 = (p1 >> 32 & low) ^ c1 ^ k0, p1 & low, (p0 >> 32 & low) ^ c3 ^ k1, p0 & low
        k0, k1 = k0 + 0x9E3779B9 & low, k1 + 0xBB67AE85 & low
    return c0, c1, c2, c3


def _normals(ids, step, last, seed):
    """Four unit normals per id: 24-bit uniforms, Box-Muller on both pairs."""
    word = torch.full_like(ids, 1)
    r = _philox((ids, word * (step & 0xFFFFFFFF), word * (step >> 32), word * last), seed)
    u = [((w >> 8).double() + 0.5) / 2.0 ** 24 for w in r]
    a, b = torch.sqrt(-2 * torch.log(u[0])), torch.sqrt(-2 * torch.log(u[2]))
    t = 2 * math.pi
    return a * torch.cos(t * u[1]), a * torch.sin(t * u[1]), b * torch.cos(t * u[3]), b * torch.sin(t * u[3])


def _mode_basis():
    x, y, z = C.T.astype(np.float64)
    c2 = x * x + y * y + z * z
    e = np.array([np.ones(19), x, y, z, c2 - 1, 3 * x * x - c2, y * y - z * z, x * y, y * z, z * x,
                  (3 * c2 - 5) * x, (3 * c2 - 5) * y, (3 * c2 - 5) * z, (y * y - z * z) * x, (z * z - x * x) * y,
                  (x * x - y * y) * z, 3 * c2 * c2 - 6 * c2 + 1, (2 * c2 - 3) * (3 * x * x - c2),
                  (2 * c2 - 3) * (y * y - z * z)])
    return e, (e * e * W).sum(axis=1)


class Exact:
    """The coupled model on one lattice: f [2, 19, nz, ny, nx], x and v [n, 3], all FP64."""

    def __init__(self, dims, m, rho, u=None, parts=None, mrt=False, substeps=1, seed=0):
        self.dims, self.m, self.mrt, self.K, self.seed, self.steps = dims, m, mrt, substeps, seed, 0
        dev = torch.device("cuda")
        self.c = torch.tensor(C, dtype=torch.float64, device=dev)
        self.w = torch.tensor(W, dtype=torch.float64, device=dev)
        shape = tuple(dims[::-1])
        u = torch.zeros((3,) + shape, dtype=torch.float64, device=dev) if u is None else u
        self.f = torch.stack([self.equilibrium(r, u) for r in rho])
        self.box = torch.tensor(dims, dtype=torch.float64, device=dev)
        self.n = 0
        if parts is not None:
            x, v, bonds, q = parts
            self.x, self.v = torch.tensor(x, device=dev), torch.tensor(v, device=dev)
            self.bonds = None if bonds is None else torch.tensor(bonds, device=dev).long()
            self.q = None if q is None else torch.tensor(q, device=dev)
            self.n = len(x)
            self.total = torch.zeros_like(self.x)

    def along(self, vec):
        """c_i . vec for every direction: [19, nz, ny, nx]."""
        return (self.c @ vec.reshape(3, -1)).reshape((19,) + tuple(vec.shape[1:]))

    def equilibrium(self, rho, u):
        cu = self.along(u)
        return self.w.view(19, 1, 1, 1) * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * (u * u).sum(0))

    def moments(self):
        rho = self.f.sum(1)
        j = (self.c.T @ self.f.sum(0).reshape(19, -1)).reshape((3,) + tuple(rho.shape[1:]))
        return rho, j

    def stencil(self, rho):
        s = torch.zeros((3,) + tuple(rho.shape), dtype=torch.float64, device=rho.device)
        for i in range(1, 19):
            r = W[i] * torch.roll(rho, tuple(-int(k) for k in C[i][::-1]), (0, 1, 2))
            for a in range(3):
                if C[i][a]:
                    s[a] += int(C[i][a]) * r
        return s

    def corners(self, x):
        """Node index and trilinear weight of the 8 corners of each cell, and x - corner: [n, 8(, 3)]."""
        cell = torch.floor(x)
        o = torch.tensor([(k & 1, k >> 1 & 1, k >> 2 & 1) for k in range(8)], dtype=torch.float64, device=x.device)
        d = (x - cell)[:, None] - o
        node = (cell[:, None] + o).remainder(self.box).long()
        return (node[..., 2] * self.dims[1] + node[..., 1]) * self.dims[0] + node[..., 0], (1 - d.abs()).prod(2), d

    def nearest(self, d):
        return d - self.box * torch.round(d / self.box)

    def pair_forces(self, x):
        force, (eps, sigma) = torch.zeros_like(x), self.m["wca"]
        for i in range(0, self.n, 1000):
            d = self.nearest(x[i:i + 1000, None] - x[None])
            r2 = (d * d).sum(2)
            r2[torch.arange(r2.shape[0]), torch.arange(i, i + r2.shape[0])] = math.inf
            s6 = (sigma * sigma / r2) ** 3
            scale = torch.where(r2 < 2 ** (1 / 3) * sigma * sigma, 24 * eps * (2 * s6 * s6 - s6) / r2, 0.0)
            if self.m["dh"]:
                lB, kappa, rc = self.m["dh"]
                r = torch.sqrt(r2)
                yukawa = lB * torch.exp(-kappa * r) * (1 / r2 + kappa / r) / r
                scale = scale + torch.where(r2 < rc * rc, self.q[i:i + 1000, None] * self.q * yukawa, 0.0)
            force[i:i + 1000] = (scale[..., None] * d).sum(1)
        if self.bonds is not None:
            k, r0 = self.m["fene"]
            d = self.nearest(x[self.bonds[:, 0]] - x[self.bonds[:, 1]])
            one = -k / (1 - (d * d).sum(1, keepdim=True) / (r0 * r0)) * d
            force.index_add_(0, self.bonds[:, 0], one).index_add_(0, self.bonds[:, 1], -one)
        return force

    def geometry(self, d):
        """sum over the 18 neighbours of Theta(d.c / |d||c|) c / |c|^2, Theta = 1 strictly inside (0, 1)."""
        c = self.c[1:]
        parallel = (torch.linalg.cross(d[..., None, :].expand(*d.shape[:-1], 18, 3),
                                       c.expand(*d.shape[:-1], 18, 3)) == 0).all(-1)
        use = ((d @ c.T > 0) & ~parallel).double()
        return use @ (c / (c * c).sum(1, keepdim=True))

    def particles(self, rho, j, S, G):
        """Advances the particles by one lattice step; adds their forces on the fluid to G [2, 3, N]."""
        m, N, K = self.m, rho[0].numel(), self.K
        r, lam = rho.reshape(2, N), m["lam"]
        fs = torch.zeros_like(G)
        own = torch.zeros_like(self.x)
        if any(lam):
            node, _, d = self.corners(self.x)
            geo = self.geometry(d)
            for z in range(2):
                push = -lam[z] * r[z][node][..., None] * geo
                fs[z].index_add_(1, node.ravel(), push.reshape(-1, 3).T)
                own -= push.sum(1)
        ucpl = (j.reshape(3, N) + 0.5 * (G + fs).sum(0)) / r.sum(0)
        G += fs
        share = r / r.sum(0)
        dt = 1.0 / K
        ids = torch.arange(self.n, device=self.x.device)
        for sub in range(K):
            node, w, _ = self.corners(self.x)
            at = lambda field: (w[..., None] * field.reshape(3, N).T[node]).sum(1)  # noqa: E731
            noise = torch.stack(_normals(ids, self.steps * K + sub, 0x4C42, self.seed)[:3], 1)
            fric = -m["gamma"] * (self.v - at(ucpl)) + math.sqrt(2 * m["kT"] * m["gamma"] / dt) * noise
            ps = [-3 * m["kappa"][z] * at(S[z]) for z in range(2)]
            for z in range(2):
                back = -share[z][node][..., None] * fric[:, None] - ps[z][:, None]
                G[z].index_add_(1, node.ravel(), (w[..., None] * back / K).reshape(-1, 3).T)
            self.total = fric + ps[0] + ps[1] + own + self.pair_forces(self.x)
            self.v = self.v + self.total * dt / m["mass"]
            self.x = (self.x + self.v * dt).remainder(self.box)

    def step(self):
        m, shape = self.m, self.f.shape[2:]
        rho, j = self.moments()
        S = [self.stencil(r) for r in rho]
        G = torch.stack([-m["g"] * rho[0] * S[1], -m["g"] * rho[1] * S[0]]).reshape(2, 3, -1)
        if self.n:
            self.particles(rho, j, S, G)
        del S
        G = G.reshape((2, 3) + tuple(shape))
        u = (j + 0.5 * G.sum(0)) / rho.sum(0)
        cu = self.along(u)
        w = self.w.view(19, 1, 1, 1)
        if self.mrt:
            noise = self.fluid_noise(rho)
        for z in range(2):
            feq = self.equilibrium(rho[z], u)
            cg, ug = self.along(G[z]), (u * G[z]).sum(0)
            source = w * 3 * (0.5 * cg + 1.5 * cu * cg - 0.5 * ug)  # every eigenvalue -1/tau = -1
            post = feq + source  # tau = 1: f* = f^eq + source
            if self.mrt:
                post = post + noise[z]
            for i in range(19):
                self.f[z, i] = torch.roll(post[i], tuple(int(k) for k in C[i][::-1]), (0, 1, 2))
        self.steps += 1

    def fluid_noise(self, rho):
        """The noise of the modes, back in the populations: [2, 19, nz, ny, nx] (eigenvalues -1)."""
        e, b = _mode_basis()
        e, b = torch.tensor(e, device="cuda"), torch.tensor(b, device="cuda")
        shape, N, kT = rho.shape[1:], rho[0].numel(), self.m["kT"]
        ids = torch.arange(N, device="cuda")
        normal = [n for k in range(9) for n in _normals(ids, self.steps, 0x464C0000 + k, self.seed)]
        r = rho.reshape(2, N)
        out = []
        for z in range(2):
            f = torch.zeros((19, N), dtype=torch.float64, device="cuda")
            for k in range(1, 19):
                if k <= 3:
                    mode = (1 if z == 0 else -1) * torch.sqrt(kT * r[0] * r[1] / r.sum(0)) * normal[k - 1]
                else:
                    mode = torch.sqrt(3 * kT * b[k] * r[z]) * normal[3 + 15 * z + k - 4]
                f += (self.w * e[k] / b[k])[:, None] * mode
            out.append(f.reshape((19,) + tuple(shape)))
        return out


def exact(case, seed):
    if case["kind"] == "replicas":
        return None  # thousands of small steps one after another
    sites = math.prod(_dims(case))
    if sites * case.get("steps", 1) > 250_000_000:
        return None
    rho = [torch.tensor(r, dtype=torch.float64, device="cuda") for r in _densities(case, seed)]
    parts = _particles(case, seed)
    if case["kind"] == "observe":
        u = torch.tensor(_flow(case, seed), dtype=torch.float64, device="cuda").permute(3, 0, 1, 2)
        e = Exact(_dims(case), _model(case), rho, u, seed=seed)
        density, j = e.moments()
        G = -e.m["g"] * (density[0] * e.stencil(density[1]) + density[1] * e.stencil(density[0]))
        velocity = (j + 0.5 * G) / density.sum(0)
        moving = [0.0] * 3 if parts is None else (e.m["mass"] * parts[1].sum(axis=0)).tolist()
        totals = torch.tensor([float(t) for t in density.sum((1, 2, 3))] + [float(t) for t in j.sum((1, 2, 3))] + moving,
                              dtype=torch.float64)
        return {"totals": totals, "rho_A": density[0], "rho_B": density[1], "u": velocity.permute(1, 2, 3, 0)}
    e = Exact(_dims(case), _model(case), rho, parts=parts, mrt=case["collision"] == "mrt", substeps=case["substeps"],
              seed=seed)
    del rho
    for _ in range(case["steps"]):
        e.step()
    out = {"f_A": e.f[0], "f_B": e.f[1]}
    if e.n:
        out.update(x=e.x, v=e.v, force=e.total)
    return out
