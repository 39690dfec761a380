"""The work that a user of the library has it do, as cases to be timed.

Every case is a simulation as a program runs it: a box (or a batch of boxes, or
a mixture of several species) is set up from host densities once, and a pass
advances it by some steps and takes from it what such a program takes: the
populations in its own device buffer, the fields on the host, or a structure
factor or interface spectrum.  The sizes are those of this repository's
benchmark, tests and design notes, and of the paper's Sec. VI.

``exact`` evaluates the same pass in 64 bits with torch alone: the lattice
update of Sec. V B written with dense moment matrices, the counter-based noise
of the library's interface (Philox4x32-10, six 21-bit uniforms a block,
Box-Muller) and the observables' definitions.
"""
from __future__ import annotations

import math

import numpy as np
import torch

KINDS = ("box", "fields", "sk", "capillary", "batch", "species")
BYTES = {"f32": 4, "f16": 2, "bf16": 2}
DTYPE = {"f32": torch.float32, "f16": torch.float16, "bf16": torch.bfloat16}


def _case(name, kind, lattice, nx, ny, nz, steps, **more):
    c = dict(name=name, kind=kind, lattice=lattice, nx=nx, ny=ny, nz=nz, steps=steps, storage="f32",
             streaming="two_arrays", schedule="two_kernels", graph_steps=0, tau_a=1.0, tau_b=1.0, kT=1e-5, G=0.9)
    c.update(more)
    return c


def listed():
    return [
        # the benchmark's workload and its 20 timed steps: the largest 3D mixture, default settings
        _case("mixture_256", "box", "D3Q19", 256, 256, 256, 20),
        # the same mixture end to end, as the benchmark's e2e figure: densities from the host, fields back to it
        _case("mixture_fields", "fields", "D3Q19", 192, 160, 144, 20),
        # 16-bit population storage, which halves the memory of a large box
        _case("mixture_bf16", "box", "D3Q19", 192, 192, 192, 20, storage="bf16"),
        # two different relaxation times (the general collision) on a box of odd sides
        _case("mixture_two_taus", "box", "D3Q19", 161, 150, 133, 10, tau_a=0.8, tau_b=1.0),
        # one population array, for boxes that fill the memory
        _case("mixture_in_place", "box", "D3Q19", 224, 200, 176, 20, streaming="in_place"),
        # the sampling loop of a structure-factor run: some steps, then one snapshot of S(k)
        _case("sampling_128", "sk", "D3Q19", 128, 128, 128, 10),
        # the largest 2D box of the benchmark, with the schedule and graphs its autotuner picks
        _case("plane_4096", "box", "D2Q9", 4096, 4096, 1, 16, schedule="tiled", graph_steps=16),
        # the 512^2 Shan-Chen box (tau = 0.8/1.0), which fits in L2 and is replayed from graphs
        _case("plane_512", "box", "D2Q9", 512, 512, 1, 160, graph_steps=16, tau_a=0.8, tau_b=1.0),
        # the capillary stripe of Sec. VI B between two height snapshots
        _case("capillary", "capillary", "D2Q9", 100, 512, 1, 256, graph_steps=64, G=1.5),
        # the ensemble of 64 small boxes of uneven size advanced together
        _case("batch_64", "batch", "D2Q9", 512, 512, 1, 64, schedule="tiled", graph_steps=64, replicas=64),
        # the paper's smallest box (Sec. VI A), where each call is all latency: some steps and a snapshot
        _case("paper_64x2", "sk", "D2Q9", 64, 2, 1, 10, G=0.4),
        # three species of different relaxation times (App. C-D), stepped between two looks at the fields
        _case("three_species", "species", "D3Q19", 96, 96, 96, 100, species=3, tau_a=0.8),
    ]


def _between(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same kinds: sizes (odd ones included) spread over the logarithm of their range."""
    kind = rng.choice(("box", "box", "box", "box", "fields", "sk", "capillary", "batch", "species"))
    two = rng.random() < 0.5
    c = dict(tau_a=0.8, tau_b=1.0) if two else {}
    c["kT"] = 10.0 ** rng.uniform(-6.0, -4.0)
    c["G"] = rng.uniform(0.0, 0.9)
    if kind == "capillary":
        c = dict(kT=10.0 ** rng.uniform(-6.0, -5.0), G=1.5, graph_steps=rng.choice((16, 64)))
        out = _case("", kind, "D2Q9", _between(rng, 80, 256), _between(rng, 64, 1024), 1, 2 * _between(rng, 16, 256), **c)
    elif kind == "batch":
        c.update(schedule=rng.choice(("tiled", "two_kernels")), graph_steps=rng.choice((16, 64)),
                 replicas=_between(rng, 4, 64))
        out = _case("", kind, "D2Q9", 512, 512, 1, 2 * _between(rng, 8, 64), **c)
    elif kind == "species":
        c["species"] = rng.choice((2, 3, 4))
        out = _case("", kind, "D3Q19", _between(rng, 24, 128), _between(rng, 24, 128), _between(rng, 24, 128),
                    2 * _between(rng, 1, 50), **c)
    elif kind == "box" and rng.random() < 0.4:
        c["graph_steps"] = rng.choice((0, 16, 64))
        c["schedule"] = rng.choice(("tiled", "two_kernels"))
        out = _case("", kind, "D2Q9", _between(rng, 64, 4096), _between(rng, 64, 4096), 1, 2 * _between(rng, 4, 80), **c)
    else:
        c["storage"] = rng.choice(("f32", "f32", "f16", "bf16")) if kind == "box" else "f32"
        c["streaming"] = rng.choice(("two_arrays", "two_arrays", "in_place"))
        side = [_between(rng, 24, 256) for _ in range(3)]
        out = _case("", kind, "D3Q19", side[0], side[1], side[2], 2 * _between(rng, 1, 20), **c)
    del out["name"]
    # no more work than the largest listed case
    most = 256 ** 3 * 20 if out["lattice"] == "D3Q19" else 4096 ** 2 * 16
    sites = out["nx"] * out["ny"] * out["nz"] if kind != "batch" else 262144 * out["replicas"]
    out["steps"] = max(2, min(out["steps"], 2 * (most // (2 * sites))))
    return out


# ---------------------------------------------------------------------------
# what a program has in hand, and one pass
# ---------------------------------------------------------------------------
_stream = None


def _one_stream():
    """A program that runs its boxes one after the other keeps them on one stream."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return _stream


def _noise_key(seed):
    return 1 + (int(seed) * 2654435761) % (2 ** 61)


def _densities(case, seed):
    """Host densities [species][z][y][x]: rho0 plus a small random part, float values held as doubles.  The
    capillary box holds a stripe rich in the first species instead."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    shape = (case["nz"], case["ny"], case["nx"])
    ns = case.get("species", 2)
    if case["kind"] == "capillary":
        nx = case["nx"]
        x = torch.arange(nx, device="cuda", dtype=torch.float64).expand(shape)
        phi = 0.25 * (1 + torch.tanh((x - 0.25 * nx) / 2.0)) * (1 - torch.tanh((x - 0.75 * nx) / 2.0))
        base = torch.stack([0.06 + 2.24 * phi, 0.06 + 2.24 * (1 - phi)])
    else:
        base = torch.tensor(_rho0(case), device="cuda", dtype=torch.float64).view(ns, 1, 1, 1).expand((ns,) + shape)
    rho = base + 1e-3 * base * torch.randn((ns,) + shape, generator=g, device="cuda", dtype=torch.float64)
    return rho.float().double().cpu().numpy()


def _rho0(case):
    if case["kind"] == "species":
        return [1.0, 0.75, 0.625, 0.875][:case["species"]]
    return [1.1875, 1.1875] if case["kind"] == "capillary" else [1.0, 1.0]


def _taus(case):
    if case["kind"] == "species":  # every relaxation time 1, or each species its own
        return [1.0] * case["species"] if case["tau_a"] == case["tau_b"] else [1.0, 0.8, 1.25, 0.9][:case["species"]]
    return [case["tau_a"], case["tau_b"]]


def _replicas(case, seed):
    """The batch's boxes: sides from {64, 128, 256, 512}, kT log-uniform, G uniform (the repository's recipe)."""
    from paper_1410_5584_gb300 import inputs

    cfg = inputs.batch_replica_configs(case["replicas"], 7)  # the boxes are the case's, the noise is the seed's
    return [dict(nx=c["nx"], ny=c["ny"], nz=1, tau_a=case["tau_a"], tau_b=case["tau_b"], kT=c["kT"], G=c["G"],
                 seed=_noise_key(seed) + k) for k, c in enumerate(cfg)]


def _batch_densities(case, seed, reps):
    parts = [_densities(dict(case, nx=r["nx"], ny=r["ny"], nz=1), 1000 * int(seed) + k) for k, r in enumerate(reps)]
    return parts


def _lattice(case):
    from paper_1410_5584_gb300 import D2Q9, D3Q19

    return D2Q9 if case["lattice"] == "D2Q9" else D3Q19


def prepare(case, seed):
    from paper_1410_5584_gb300 import Batch, Lattice, MultiLattice
    from paper_1410_5584_gb300 import flbm

    state = dict(case=case)
    if case["kind"] == "batch":
        reps = _replicas(case, seed)
        b = Batch(_lattice(case), reps, storage=case["storage"], stream=_one_stream(),
                  schedule=flbm.SCHEDULE[case["schedule"]], graph_steps=case["graph_steps"])
        rho = _batch_densities(case, seed, reps)
        b.init(np.concatenate([r[0].ravel() for r in rho]), np.concatenate([r[1].ravel() for r in rho]))
        state.update(sim=b)
    elif case["kind"] == "species":
        ns = case["species"]
        G = 0.3 * (1.0 - np.eye(ns))
        m = MultiLattice(_lattice(case), ns, case["nx"], case["ny"], case["nz"], tau=_taus(case), kT=case["kT"], G=G,
                         seed=_noise_key(seed), rho0=_rho0(case), stream=_one_stream(), streaming=case["streaming"])
        m.init(_densities(case, seed))
        state.update(sim=m)
    else:
        r0 = _rho0(case)
        lat = Lattice(_lattice(case), case["nx"], case["ny"], case["nz"], case["tau_a"], case["tau_b"], case["kT"],
                      case["G"], seed=_noise_key(seed), storage=case["storage"], stream=_one_stream(),
                      streaming=flbm.STREAMING[case["streaming"]], schedule=flbm.SCHEDULE[case["schedule"]],
                      graph_steps=case["graph_steps"], rho0_a=r0[0], rho0_b=r0[1])
        rho = _densities(case, seed)
        if case["kind"] == "fields":
            state.update(rho=rho)
        else:
            lat.init(rho[0], rho[1])
        state.update(sim=lat)
    if case["kind"] in ("box", "sk", "capillary", "batch"):
        # the current populations after an even number of steps: the first array of the context's buffer
        n = 2 * state["sim"].Q * state["sim"].N
        state["pop"] = state["sim"].pop_buffer.view(DTYPE[case["storage"]])[:n]
    return state


def run(state):
    case, sim = state["case"], state["sim"]
    kind = case["kind"]
    if kind == "fields":
        sim.init(state["rho"][0], state["rho"][1])
        sim.step(case["steps"])
        return sim.moments()
    sim.step(case["steps"])
    if kind == "species":
        return sim.moments()
    if kind == "sk":
        sim.sf_sample()
        return [state["pop"], *sim.structure_factor(0)[:4]]
    if kind == "capillary":
        sim.cap_sample(-1, -1)
        return [state["pop"], *sim.cap_spectrum()[:2]]
    return [state["pop"]]


def work(case):
    """Populations read and written once a pass, plus what crosses to and from the host; about 40 operations a
    step for each population (transforms, force, equilibrium, noise)."""
    q = 9 if case["lattice"] == "D2Q9" else 19
    d = 2 if case["lattice"] == "D2Q9" else 3
    ns = case.get("species", 2)
    if case["kind"] == "batch":
        sites = sum(r["nx"] * r["ny"] for r in _replicas(case, 0))
    else:
        sites = case["nx"] * case["ny"] * case["nz"]
    moved = 2 * ns * q * BYTES[case["storage"]] * sites
    if case["kind"] == "fields":
        moved = (2 * 8 + (2 + d) * 8) * sites  # densities in, fields out: no populations are asked for
    elif case["kind"] == "species":
        moved += (ns + d) * 8 * sites
    return {"bytes": moved, "flops": 40 * ns * q * sites * case["steps"]}


# ---------------------------------------------------------------------------
# the same pass in 64 bits
# ---------------------------------------------------------------------------
def _basis(lattice):
    """Velocities, weights, moment rows and norms (D2Q9: Table I of the paper; D3Q19: the interface's basis)."""
    if lattice == "D2Q9":
        c = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
        w = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4
        c = [(x, y, 0) for x, y in c]
        def rows(x, y, z):
            s = x * x + y * y
            return [1, x, y, 3 * s - 2, 2 * x * x - s, x * y, (3 * s - 4) * x, (3 * s - 4) * y, 9 * s * s - 15 * s + 2]
        d = 2
    else:
        c = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
             (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
             (0, -1, 1)]
        w = [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12
        def rows(x, y, z):
            s = x * x + y * y + z * z
            return [1, x, y, z, s - 1, 2 * x * x - y * y - z * z, y * y - z * z, x * y, y * z, x * z, (3 * s - 5) * x,
                    (3 * s - 5) * y, (3 * s - 5) * z, x * (y * y - z * z), y * (z * z - x * x), z * (x * x - y * y),
                    3 * s * s - 6 * s + 1, (2 * s - 3) * (2 * x * x - y * y - z * z), (2 * s - 3) * (y * y - z * z)]
        d = 3
    T = np.array([rows(*v) for v in c], dtype=np.float64).T  # [mode][i]
    w = np.array(w)
    return d, c, w, T, (T * T * w).sum(1)


def _philox(site, step, species, block, key):
    """The four output words of Philox4x32-10 for counter (site, step, species, block); int64 tensors of 32-bit words."""
    mask = 0xFFFFFFFF
    x = [site, torch.full_like(site, step & mask), torch.full_like(site, species), torch.full_like(site, block)]
    k0, k1 = key & mask, (key >> 32) & mask
    for _ in range(10):
        p0, p1 = x[0] * 0xD2511F53, x[2] * 0xCD9E8D57  # 64-bit products modulo 2^64
        x = [((p1 >> 32) & mask) ^ x[1] ^ k0, p1 & mask, ((p0 >> 32) & mask) ^ x[3] ^ k1, p0 & mask]
        k0, k1 = (k0 + 0x9E3779B9) & mask, (k1 + 0xBB67AE85) & mask
    return x


def _gaussians(q, site, step, species, key):
    """[mode] unit Gaussians of one species; mode a is Gaussian a - 1 of its blocks of six."""
    g = [None] * q
    for b in range((q + 4) // 6):
        x = _philox(site, step, species, b, key)
        u = [v >> 11 for v in x] + [((x[0] & 0x7FF) << 10) + (x[1] & 0x3FF), ((x[2] & 0x7FF) << 10) + (x[3] & 0x3FF)]
        for p in range(3):
            a = 6 * b + 2 * p + 1
            if a >= q:
                break
            r = torch.sqrt(-2.0 * torch.log((u[2 * p] + 1).double() * 2.0 ** -21))
            t = u[2 * p + 1].double() * (2.0 * math.pi * 2.0 ** -21)
            g[a] = r * torch.cos(t)
            if a + 1 < q:
                g[a + 1] = r * torch.sin(t)
    return g


class _Exact:
    """Boxes of one shape advanced together in 64 bits: f[species][i] is a tensor [box][z][y][x]."""

    def __init__(self, lattice, rho, taus, kT, G, keys, shared):
        self.d, self.c, w, T, norms = _basis(lattice)
        self.q, self.ns = len(self.c), len(taus)
        dev = dict(device="cuda", dtype=torch.float64)
        self.w, self.T, self.norms = w, torch.tensor(T, **dev), norms
        self.rho0 = None
        nb, (nz, ny, nx) = len(keys), rho.shape[2:]
        self.shape = (nb, nz, ny, nx)
        self.site = torch.arange(nz * ny * nx, device="cuda").view(1, nz, ny, nx)
        self.f = [torch.stack([rho[s] * w[i] for i in range(self.q)]) for s in range(self.ns)]
        per_box = lambda v: torch.tensor(v, **dev).view(nb, 1, 1, 1)  # noqa: E731
        self.kT, self.G = per_box(kT), G  # G[s][t]: a tensor over the boxes, or a number
        self.keys, self.shared, self.step_no = keys, shared, 0
        self.rate = [1.0 / t for t in taus]
        self.rate_d = (1.0 / taus[0] if len(set(taus)) == 1 else len(taus) / sum(taus))
        # projections of a second-order Hermite tensor Q_ab on the modes
        cs2 = 1.0 / 3.0
        self.second = {}
        for a in range(self.d):
            for b in range(a, self.d):
                h = np.array([v[a] * v[b] - (cs2 if a == b else 0.0) for v in self.c]) * w / (2 * cs2 * cs2)
                self.second[a, b] = (T @ h) * (1.0 if a == b else 2.0)

    def shift(self, field, v):
        """field at r + v."""
        return torch.roll(field, (-v[2], -v[1], -v[0]), (-3, -2, -1))

    def density_and_force(self):
        rho = [f.sum(0) for f in self.f]
        grad = []
        for s in range(self.ns):
            g = [torch.zeros_like(rho[s]) for _ in range(self.d)]
            for i in range(1, self.q):
                n = self.shift(rho[s], self.c[i])
                for a in range(self.d):
                    if self.c[i][a]:
                        g[a] += self.w[i] * self.c[i][a] * n
            grad.append(g)
        acc = [[-sum(self.G[s][t] * grad[t][a] for t in range(self.ns) if t != s) for a in range(self.d)]
               for s in range(self.ns)]
        return rho, acc

    def project(self, pairs):
        """sum_ab second[a, b] Q_ab as {mode: tensor} of the modes it reaches."""
        out = {}
        for (a, b), q in pairs.items():
            for m in range(self.d + 1, self.q):
                k = self.second[a, b][m]
                if abs(k) > 1e-12:
                    out[m] = out[m] + k * q if m in out else k * q
        return out

    def noise(self, rho, rt):
        """Momentum noise [species][axis] and the unit Gaussians [species][mode] of every box."""
        g = [[None] * self.q for _ in range(self.ns)]
        for s in range(self.ns):
            per = [_gaussians(self.q, self.site, self.step_no, s, k) for k in self.keys]
            for a in range(1, self.q):
                g[s][a] = torch.cat([p[a] for p in per], 0)
            del per
        amp = torch.sqrt((2 * self.rate_d - self.rate_d ** 2) * self.kT)
        xi = [[None] * self.d for _ in range(self.ns)]
        for a in range(self.d):
            if self.shared:
                v = amp * torch.sqrt(rho[0] * rho[1] / rt) * g[0][a + 1]
                xi[0][a], xi[1][a] = v, -v
            else:
                tot = sum(torch.sqrt(rho[s]) * g[s][a + 1] for s in range(self.ns)) / rt
                for s in range(self.ns):
                    xi[s][a] = amp * (torch.sqrt(rho[s]) * g[s][a + 1] - rho[s] * tot)
        return xi, g

    def moment(self, s, m):
        """m_a of one species, the zero entries of its row left out."""
        out = None
        for i in range(self.q):
            t = float(self.T[m, i])
            if t:
                out = t * self.f[s][i] if out is None else out + t * self.f[s][i]
        return out

    def step(self):
        rho, acc = self.density_and_force()
        rt = sum(rho)
        j = [[self.moment(s, 1 + a) for a in range(self.d)] for s in range(self.ns)]
        u = [sum(j[s][a] + 0.5 * rho[s] * acc[s][a] for s in range(self.ns)) / rt for a in range(self.d)]
        xi, g = self.noise(rho, rt)
        ld = self.rate_d
        axes = [(a, b) for a in range(self.d) for b in range(a, self.d)]
        for s in range(self.ns):
            R = [ld * (rho[s] * u[a] - j[s][a]) + (1 - ld / 2) * rho[s] * acc[s][a] + xi[s][a] for a in range(self.d)]
            v = [(j[s][a] + 0.5 * R[a]) / rho[s] for a in range(self.d)]
            eq = self.project({(a, b): rho[s] * u[a] * u[b] for a, b in axes})
            phi = self.project({(a, b): rho[s] * (acc[s][a] * v[b] + v[a] * acc[s][b]) for a, b in axes})
            lb = self.rate[s]
            add = {1 + a: R[a] / self.norms[1 + a] for a in range(self.d)}
            for m in range(self.d + 1, self.q):
                change = torch.sqrt((2 * lb - lb * lb) * 3.0 * self.kT * self.norms[m] * rho[s]) * g[s][m]
                change = change - lb * self.moment(s, m)
                if m in eq:
                    change += lb * eq[m] + (1 - lb / 2) * phi[m]
                add[m] = change / self.norms[m]
                g[s][m] = None
            new = torch.empty_like(self.f[s])
            for i in range(self.q):
                y = self.f[s][i].clone()
                for m, t in add.items():
                    k = float(self.T[m, i])
                    if k:
                        y += (self.w[i] * k) * t
                v_ = self.c[i]
                new[i] = torch.roll(y, (v_[2], v_[1], v_[0]), (-3, -2, -1))
            self.f[s] = new
        self.step_no += 1

    def velocity(self):
        rho, acc = self.density_and_force()
        rt = sum(rho)
        j = [sum(self.moment(s, 1 + a) + 0.5 * rho[s] * acc[s][a] for s in range(self.ns)) for a in range(self.d)]
        return rho, j, [v / rt for v in j]

    def populations(self, box, rho0):
        """The device layout of one box: [i][site][species] deviations from w_i rho0."""
        parts = [torch.stack([self.f[s][i, box] - self.w[i] * rho0[s] for i in range(self.q)]).view(self.q, -1)
                 for s in range(self.ns)]
        return torch.stack(parts, -1).reshape(-1)


def _exact_boxes(case, rho, kT, G, keys):
    """rho: [species][box][z][y][x]."""
    two = case["kind"] != "species"
    dev = dict(device="cuda", dtype=torch.float64)
    if two:
        g = torch.tensor(G, **dev).view(len(keys), 1, 1, 1)
        coupling = [[0.0, g], [g, 0.0]]
    else:
        coupling = [[0.0 if s == t else 0.3 for t in range(case["species"])] for s in range(case["species"])]
    sim = _Exact(case["lattice"], torch.tensor(rho, **dev), _taus(case), kT, coupling, keys, two)
    for _ in range(case["steps"]):
        sim.step()
    return sim


def _exact_sk(sim):
    rho, _, u = sim.velocity()
    n, nx = sim.site.numel(), sim.shape[3]
    spec = lambda v: torch.fft.fft(v[0].sum((0, 1)))[1:nx // 2 + 1]  # noqa: E731
    a, b, us = spec(rho[0]), spec(rho[1]), [spec(v) for v in u]
    S_uu = sum(v.abs().square() for v in us) / (sim.d * n)
    return [a.abs().square() / n, (a * b.conj()).real / n, b.abs().square() / n, S_uu]


def _exact_heights(sim):
    """Spectrum and mean heights of a stripe's two interfaces, the columns tracked as the interface documents."""
    r = sim.f[0].sum(0)[0, 0].cpu().numpy()  # [y][x]
    ny, nx = r.shape
    col = (r - 1.1875).sum(0)
    window = np.array([np.take(col, range(x, x + nx // 2), mode="wrap").sum() for x in range(nx)])
    xl = (int(np.argmax(window)) + nx // 2 // 2) % nx
    xg = (xl + nx // 2) % nx
    rl, rg = r[:, xl].mean(), r[:, xg].mean()
    frac = (r - rg) / (rl - rg)
    n1 = (xl - xg) % nx
    L1 = np.take(frac, range(xg, xg + n1), axis=1, mode="wrap").sum(1)
    L2 = np.take(frac, range(xl, xl + nx - n1), axis=1, mode="wrap").sum(1)
    h = np.stack([xl - 0.5 - L1, xl - 0.5 + L2])
    spec = np.abs(np.fft.fft(h - h.mean(1, keepdims=True), axis=1)) ** 2 / ny
    return [spec.mean(0)[1:ny // 2 + 1], h.mean(1)]


def exact(case, seed):
    if case["kind"] == "batch":
        reps = _replicas(case, seed)
        rho = _batch_densities(case, seed, reps)
        by_shape = {}
        for k, r in enumerate(reps):
            by_shape.setdefault((r["ny"], r["nx"]), []).append(k)
        parts = [None] * len(reps)
        for ks in by_shape.values():
            sim = _exact_boxes(case, np.stack([rho[k] for k in ks], 1), [reps[k]["kT"] for k in ks],
                               [reps[k]["G"] for k in ks], [reps[k]["seed"] for k in ks])
            for b, k in enumerate(ks):
                parts[k] = sim.populations(b, [1.0, 1.0])
        return [torch.cat(parts)]
    sim = _exact_boxes(case, _densities(case, seed)[:, None], [case["kT"]], [case["G"]], [_noise_key(seed)])
    if case["kind"] in ("fields", "species"):
        rho, j, u = sim.velocity()
        cons = [float(r.sum()) for r in rho] + [float(v.sum()) for v in j]
        fields = [r[0].cpu().numpy() for r in rho]
        fields = fields if case["kind"] == "fields" else [np.stack(fields)]
        return (*fields, np.stack([v[0].cpu().numpy() for v in u]), np.array(cons))
    pop = sim.populations(0, _rho0(case))
    if case["kind"] == "sk":
        return [pop, *_exact_sk(sim)]
    if case["kind"] == "capillary":
        return [pop, *_exact_heights(sim)]
    return [pop]
