"""Performance cases of the FETD-PIC framework: what its users have it do, timed through its public
entry points.

A pass advances a simulation by one diagnostic interval (`steps` time steps) and hands back the state
the program then looks at: particle positions and momenta, the field unknowns and the current.  The
FP32 mode keeps its particles in single precision, so its programs keep their snapshots in single
precision too; the FP64 mode returns what it computed.  A state evolves from pass to pass, as a run
does.

`exact` repeats a pass in plain FP64 tensor operations: the same leapfrog (Faraday, gather, push, move,
walk, deposit, Ampere with the level-2 sparse approximate inverse), one operation at a time over all
particles, from the method's equations.
"""
import functools
import math

import numpy as np
import torch

from paper_1707_04333_gb300 import fetdpic, inputs

C = inputs.C_LIGHT
Q_E, M_E, EPS0, MU0 = inputs.Q_E, inputs.M_E, inputs.EPS0, inputs.MU0
# electrons per superparticle of the beam and cyclotron runs: their field stands clear of the applied
# field's rounding and is still too weak to move them
WEIGHT = 1e6


def listed():
    return [
        # RF-driven acceleration of a single electron: the drive's amplitude follows the electron, so
        # every step is a call of its own with a read behind it.  The smallest calls: latency only.
        dict(name="rf_electron", kind="rf", nx=100, steps=8, pusher="boris", precision="fp64"),
        # Gyro-orbit precision run: 64 superparticles on the 2,048-triangle square, thousands of steps with
        # a look every 256: launches and their gaps.
        dict(name="cyclotron_64", kind="cyclotron", nx=32, n=64, gamma=2.0, steps=256, pusher="boris", precision="fp32"),
        # The Bernstein-mode strip, periodic top and bottom, with its line of field probes.
        dict(name="bernstein_strip", kind="pair", nx=1024, ny=4, ppc=20, kT=0.05, ratio=1.0 / 3.0, steps=128,
             pusher="vay", precision="fp32", probes=256),
        # The same kind of run on the plain FP64 path, which FP32 results are judged against.
        dict(name="pair_8k_fp64", kind="pair", nx=64, ny=64, ppc=20, kT=0.1, ratio=0.5, steps=64, pusher="vay",
             precision="fp64"),
        # FP64 at a size that fills the chip, with the volume-preserving pusher.
        dict(name="pair_51k_fp64", kind="pair", nx=160, ny=160, ppc=20, kT=0.1, ratio=0.5, steps=16, pusher="hc",
             precision="fp64"),
        # The benchmark's pair plasma: 200,978 triangles, 8.04 M particles.
        dict(name="pair_200k", kind="pair", nx=317, ny=317, ppc=20, kT=0.1, ratio=0.5, steps=128, pusher="vay",
             precision="fp32"),
        # A fine mesh with few particles, where the field update is the larger half of a step.
        dict(name="sparse_320k", kind="pair", nx=400, ny=400, ppc=1, kT=0.02, ratio=0.7, steps=64, pusher="boris",
             precision="fp32"),
        # Parameter sweep: independent uneven plasmas in one context.
        dict(name="batched_16", kind="batch", instances=16, f_lo=2000, f_hi=50000, p_lo=4000, p_hi=400000, steps=32,
             pusher="vay", precision="fp32"),
        # High-gamma beam in crossed applied fields: every particle above gamma = 10.
        dict(name="beam_6m", kind="beam", nx=250, n=6250000, steps=16, pusher="hc", precision="fp32"),
        # A run that watches its conservation laws every fourth step.
        dict(name="checked_20k", kind="pair", nx=101, ny=99, ppc=20, kT=0.1, ratio=0.5, steps=32, pusher="boris_tan",
             precision="fp32", check=4),
        # Particle state streamed from page-locked host memory and back every step (coupling to a host code).
        dict(name="stream_2m", kind="pair", nx=160, ny=160, ppc=20, kT=0.1, ratio=0.5, steps=1, pusher="boris",
             precision="fp32", stream=True),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _cap(particles, precision):
    """Steps that keep a drawn case below the listed ones' cost."""
    return max(4, int((6e8 if precision == "fp32" else 2.5e7) / particles))


def draw(rng):
    kind = rng.choice(["pair", "pair", "pair", "cyclotron", "batch", "beam"])
    pusher = rng.choice(["boris", "boris_tan", "vay", "hc"])
    precision = rng.choice(["fp32", "fp32", "fp64"])
    if kind == "cyclotron":
        return dict(kind=kind, nx=int(_log(rng, 16, 96)), n=int(_log(rng, 1, 4000)), gamma=rng.choice([1.1, 2.0, 10.0]),
                    steps=int(_log(rng, 64, 400)), pusher=pusher, precision=precision)
    if kind == "batch":
        n, p_hi = rng.randint(2, 20), int(_log(rng, 20000, 400000))
        steps = min(rng.randint(8, 40), _cap(n * p_hi / 3, precision))
        return dict(kind=kind, instances=n, f_lo=1000, f_hi=int(_log(rng, 4000, 50000)), p_lo=2000, p_hi=p_hi, steps=steps,
                    pusher=pusher, precision=precision)
    if kind == "beam":
        nx = int(_log(rng, 30, 200))
        return dict(kind=kind, nx=nx, n=int(2 * nx * nx * _log(rng, 4, 50)), steps=rng.randint(4, 24), pusher=pusher,
                    precision="fp32")
    nx = int(_log(rng, 16, 256))
    ny = max(6, int(nx * rng.choice([1.0, 1.0, 0.37])))
    ppc = int(_log(rng, 1, 30))
    steps = min(rng.randint(32, 96), _cap(4 * nx * ny * ppc, precision))
    case = dict(kind=kind, nx=nx, ny=ny, ppc=ppc, kT=_log(rng, 0.01, 0.3), ratio=rng.uniform(0.25, 1.0),
                steps=steps, pusher=pusher, precision=precision)
    if rng.random() < 0.25:
        case["check"] = rng.choice([1, 4, 8])
    return case


# ------------------------------------------------------------------ inputs

@functools.lru_cache(maxsize=32)
def _mesh(nx, ny, lx, ly, jitter, periodic):
    return inputs.jittered_delaunay(nx, ny, lx, ly, jitter, seed=11, periodic_y=periodic)


def _edge_lengths(mesh):
    p, t = mesh.nodes, mesh.triangles
    return np.concatenate([np.linalg.norm(p[t[:, a]] - p[t[:, b]], axis=1) for a, b in ((0, 1), (1, 2), (2, 0))])


def _in_triangles(mesh, tri, gen):
    """Uniform points in the given triangles (square-root barycentric sampling)."""
    nodes = torch.from_numpy(mesh.nodes).cuda()[torch.from_numpy(mesh.triangles).cuda().long()[tri]]
    r1 = torch.rand(len(tri), generator=gen, device="cuda", dtype=torch.float64).sqrt()
    r2 = torch.rand(len(tri), generator=gen, device="cuda", dtype=torch.float64)
    w = torch.stack([1.0 - r1, r1 * (1.0 - r2), r1 * r2], 1)
    return (w[:, :, None] * nodes).sum(1)


def _thermal(n, kT, gen):
    """In-plane momenta of a 2-D Maxwell-Juettner law: gamma - 1 is a mixture of Exp and Gamma(2)."""
    eta = 1.0 / kT
    r = torch.rand(4, n, generator=gen, device="cuda", dtype=torch.float64)
    g = -torch.log1p(-r[0]) / eta
    g = 1.0 + torch.where(r[1] < eta / (eta + 1.0), g, g - torch.log1p(-r[2]) / eta)
    p = C * torch.sqrt(g * g - 1.0)
    th = 2.0 * math.pi * r[3]
    return torch.stack([p * torch.cos(th), p * torch.sin(th)], 1)


def _np(t):
    return t.cpu().numpy()


def _pair(nx, ny, ppc, kT, ratio, pusher, periodic, gen):
    """Magnetized electron-positron plasma, collocated pairs of opposite momenta, mean edge one Debye length."""
    b0 = 5.0
    wc = Q_E * b0 / M_E
    wp = wc / ratio
    h = C * math.sqrt(kT) / wp
    mesh = _mesh(nx, ny, h * nx, h * ny, 0.3, periodic)
    nf = len(mesh.triangles)
    tri = torch.arange(nf, device="cuda").repeat_interleave(ppc)
    x, u, hint = _in_triangles(mesh, tri, gen), _thermal(nf * ppc, kT, gen), _np(tri.int())
    weight = wp * wp * EPS0 * M_E / (Q_E * Q_E) * mesh.lx * mesh.ly / (nf * ppc)
    x, u = _np(x), _np(u)
    species = [inputs.Species(-Q_E * weight, M_E * weight, x, u, hint), inputs.Species(Q_E * weight, M_E * weight, x, -u, hint)]
    dt = min(0.2 * _edge_lengths(mesh).min() / C, 0.05 / wc)
    return inputs.Workload("pair", mesh, species, dt, b0=b0, pusher=pusher)


def _workloads(case, seed):
    gen = torch.Generator("cuda")
    gen.manual_seed(seed)
    kind, pusher = case["kind"], case["pusher"]
    if kind == "pair":
        return [_pair(case["nx"], case["ny"], case["ppc"], case["kT"], case["ratio"], pusher, bool(case.get("probes")), gen)]
    if kind == "batch":
        out, n = [], case["instances"]
        for k in range(n):
            # sizes log-spaced over the sweep's range, triangles and particles in different orders
            f = math.exp(math.log(case["f_lo"]) + (k / max(1, n - 1)) * math.log(case["f_hi"] / case["f_lo"]))
            p = math.exp(math.log(case["p_lo"]) + ((k * 7) % n / max(1, n - 1)) * math.log(case["p_hi"] / case["p_lo"]))
            side = max(4, round(math.sqrt(f / 2.0)))
            kT = math.exp(math.log(0.01) + ((k * 5) % n / max(1, n - 1)) * math.log(30.0))
            out.append(_pair(side, side, max(1, round(p / (4 * side * side))), kT, 0.25 + 0.75 * k / max(1, n - 1), pusher,
                             False, gen))
        return out
    if kind == "cyclotron":
        mesh, n, g = _mesh(case["nx"], case["nx"], 1.0, 1.0, 0.3, False), case["n"], case["gamma"]
        r = torch.rand(3, n, generator=gen, device="cuda", dtype=torch.float64)
        rad, th, ph, s = 0.05 * r[0].sqrt(), 2 * math.pi * r[1], 2 * math.pi * r[2], C * math.sqrt(g * g - 1.0)
        x = torch.stack([0.5 + rad * torch.cos(th), 0.5 + rad * torch.sin(th)], 1)
        u = torch.stack([s * torch.cos(ph), s * torch.sin(ph)], 1)
        sp = inputs.Species(-Q_E * WEIGHT, M_E * WEIGHT, _np(x), _np(u), np.full(n, -1, np.int32))
        # dt of the gyration, or of the field update where the mesh is finer
        dt = min(0.05 * M_E / Q_E, 0.2 * _edge_lengths(mesh).min() / C)
        return [inputs.Workload("cyclotron", mesh, [sp], dt, b0=1.0, pusher=pusher)]
    if kind == "beam":
        side, b0 = 10.0 * case["nx"] / 707.0, 1.0
        mesh, n = _mesh(case["nx"], case["nx"], side, side, 0.3, False), case["n"]
        tri = torch.randint(len(mesh.triangles), (n,), generator=gen, device="cuda")
        x = _in_triangles(mesh, tri, gen)
        g = torch.exp(math.log(10.0) + math.log(100.0) * torch.rand(n, generator=gen, device="cuda", dtype=torch.float64))
        ux = C * torch.sqrt(g * g - 1.0)
        sp = inputs.Species(-Q_E * WEIGHT, M_E * WEIGHT, _np(x), _np(torch.stack([ux, torch.zeros_like(ux)], 1)), _np(tri.int()))
        return [inputs.Workload("beam", mesh, [sp], 0.2 * _edge_lengths(mesh).min() / C, b0=b0, ext=(0.5 * C * b0, 0.0, 0.0),
                                pusher=pusher)]
    # rf: magnet over the whole square, RF field in the gap strip; the electron's place on its first orbit varies
    w = inputs.synchrocyclotron(n=case["nx"])
    s = w.species[0]
    th = float(torch.rand(1, generator=gen, device="cuda", dtype=torch.float64)) * 0.5 - 0.25
    rot = np.array([[math.cos(th), -math.sin(th)], [math.sin(th), math.cos(th)]])
    s.x = np.ascontiguousarray((s.x - 0.5) @ rot.T + 0.5)
    s.u = np.ascontiguousarray(s.u @ rot.T)
    return [w]


class _State:
    pass


def _probe_line(mesh, n):
    """A line of points along x at mid height (a little off it, so no point lies on a mesh line)."""
    return np.stack([mesh.lx * (np.arange(n) + 0.5) / n, np.full(n, 0.4973 * mesh.ly)], 1)


def prepare(case, seed):
    s = _State()
    s.case, ws = case, _workloads(case, seed)
    single = case["precision"] == "fp32"
    check, probes = case.get("check", 0), case.get("probes", 0)
    s.sim = sim = fetdpic.Simulation(ws, precision=case["precision"], check_interval=check, use_graphs=not check)
    if probes:
        sim.set_probes(_probe_line(ws[0].mesh, probes), capacity=case["steps"])
    sim.load()
    if case["kind"] == "rf":
        s.drive = inputs.RFDrive(ws[0].ext[2], ws[0].dt, True)
        sim.read_species(0)
        return s

    # one page-locked snapshot of all species, in load order; the FP32 mode keeps a single-precision copy
    n = sum(k for _, _, k in sim.species)
    s.snap = [torch.zeros(n, 2, dtype=torch.float64, pin_memory=True), torch.zeros(n, 2, dtype=torch.float64, pin_memory=True),
              torch.zeros(n, dtype=torch.int32, pin_memory=True)]
    s.kept = [torch.zeros(n, 2, dtype=torch.float32), torch.zeros(n, 2, dtype=torch.float32)] if single else s.snap
    # the program's first look at what it loaded: the particles are on the device after it
    _snapshot(s)
    sim.sync()
    if case.get("stream"):
        s.given = [a.clone().pin_memory() for a in s.snap]
    return s


def _rows(s, arrays):
    """(species id, its rows of each array) of arrays that hold the species one after another."""
    at = 0
    for _, sid, n in s.sim.species:
        yield sid, [a[at:at + n].numpy() for a in arrays]
        at += n


def _snapshot(s):
    for sid, rows in _rows(s, s.snap):
        fetdpic.fetdpic_read_particles_async(s.sim.h, sid, *rows)


def _run_rf(s):
    sim, rows = s.sim, []
    for _ in range(s.case["steps"]):
        sim.set_external_amplitude(s.drive.amplitude())
        sim.step(1)
        got = sim.read_species(0)
        s.drive.advance(got["u"])
        rows.append(np.concatenate([got["x"][0], got["u"][0]]))
    return {"orbit": np.stack(rows), **sim.read_fields(0)}


def run(s):
    case, sim = s.case, s.sim
    if case["kind"] == "rf":
        return _run_rf(s)
    single = case["precision"] == "fp32"
    if case.get("stream"):
        for sid, rows in _rows(s, s.given):
            fetdpic.fetdpic_write_particles(sim.h, sid, *rows)
    sim.step(case["steps"], case["pusher"])
    _snapshot(s)
    sim.sync()
    if single:
        s.kept[0].copy_(s.snap[0])
        s.kept[1].copy_(s.snap[1])
    out = dict(zip(("x", "u", "cell"), s.kept))
    fields = [sim.read_fields(k) for k in range(len(sim.workloads))]
    for n in ("e", "b", "j"):
        f = np.concatenate([f[n] for f in fields]) if len(fields) > 1 else fields[0][n]
        out[n] = f.astype(np.float32) if single else f
    if case.get("probes"):
        out["probes"] = sim.read_probes()[0].astype(np.float32)
    if case.get("check"):
        # what such a run asks: is charge conserved, does Gauss's law hold, how much energy is in the field
        c = [fetdpic.fetdpic_check(sim.h, k) for k in range(len(sim.workloads))]
        out["continuity"] = all(x["dce"] < 1e-4 for x in c)
        out["gauss"] = all(x["dgl"] < 1e-4 for x in c)
        out["energy"] = [float(x["energy"]) for x in c]
    return out


def work(case):
    """State in and out once a step: particles, field unknowns, the current, the inverse's entries."""
    single = case["precision"] == "fp32"
    if case["kind"] == "pair":
        f, p = 2 * case["nx"] * case["ny"], 4 * case["nx"] * case["ny"] * case["ppc"]
    elif case["kind"] == "batch":
        n = case["instances"]
        f = sum(case["f_lo"] * (case["f_hi"] / case["f_lo"]) ** (k / max(1, n - 1)) for k in range(n))
        p = sum(case["p_lo"] * (case["p_hi"] / case["p_lo"]) ** (k / max(1, n - 1)) for k in range(n))
    else:
        f, p = 2 * case["nx"] ** 2, case.get("n", 1)
    e = 1.5 * f
    word = 4 if single else 8
    step = p * 2 * (4 + 4 * word) + f * 16 + e * (16 + 8 + 13 * (word + 4))
    given = 2 * 36 * p if case.get("stream") else 36 * p
    return {"bytes": case["steps"] * step + given + 8 * (2 * e + f), "flops": case["steps"] * (240.0 * p + 12 * f + 34 * e)}


# ------------------------------------------------- the same pass, plain FP64

class _Plain:
    """One instance of the method over FP64 tensors."""

    def __init__(self, w):
        d = torch.device("cuda")
        m = w.mesh
        self.w, self.dt = w, float(w.dt)
        xy = torch.from_numpy(m.nodes).to(d)
        tri = torch.from_numpy(m.triangles).to(d).long()
        self.nf = len(tri)
        rep = torch.arange(len(xy), device=d)
        self.period = None
        if m.periodic is not None:
            pairs = torch.from_numpy(m.periodic[0]).to(d).long()
            rep[pairs[:, 1]] = pairs[:, 0]
            self.period = torch.tensor(m.periodic[1], dtype=torch.float64, device=d)
        nxt, prv = [1, 2, 0], [2, 0, 1]
        X = xy[tri]                                              # [F, 3, 2]
        a, b = X[:, nxt], X[:, prv]
        d2a = (X[:, 1, 0] - X[:, 0, 0]) * (X[:, 2, 1] - X[:, 0, 1]) - (X[:, 2, 0] - X[:, 0, 0]) * (X[:, 1, 1] - X[:, 0, 1])
        self.inv2a, self.area = 1.0 / d2a, 0.5 * d2a
        self.grad = torch.stack([a[:, :, 1] - b[:, :, 1], b[:, :, 0] - a[:, :, 0]], 2) * self.inv2a[:, None, None]
        self.far = a                                             # lambda_m(r) = grad_m . (r - node m+1)
        # edges: sorted node pairs; local edge m runs from node m+1 to node m+2
        na, nb = rep[tri[:, nxt]], rep[tri[:, prv]]
        key = torch.minimum(na, nb) * len(xy) + torch.maximum(na, nb)
        keys, self.te = torch.unique(key, return_inverse=True)
        self.te = self.te.reshape(-1, 3)
        self.ts = torch.where(na < nb, 1.0, -1.0).double()
        self.ne = ne = len(keys)
        slot = self.te.reshape(-1)
        order = torch.argsort(slot, stable=True)
        count = torch.bincount(slot, minlength=ne)
        first = torch.cumsum(count, 0) - count
        side = torch.full((ne, 2), -1, dtype=torch.long, device=d)   # (triangle * 3 + local edge) on each side
        side[:, 0] = order[first]
        two = count > 1
        side[two, 1] = order[first[two] + 1]
        here = torch.arange(3 * self.nf, device=d)
        other = torch.where(side[slot, 0] == here, side[slot, 1], side[slot, 0])
        self.nb = torch.where(other >= 0, other, -1).reshape(-1, 3)
        self.free = torch.nonzero(two).reshape(-1)
        self.shift = torch.zeros(self.nf, 3, dtype=torch.float64, device=d)
        if self.period is not None:
            g = self.nb.clamp(min=0)
            theirs = tri[g // 3, (g % 3 + 2) % 3]
            ours = tri[:, nxt]
            self.shift = ((rep[theirs] != theirs).double() - (rep[ours] != ours).double()) * (self.nb >= 0)
        self._hodge()
        self._inverse()
        self.b = w.b0 * self.area
        self.e = torch.zeros(ne, dtype=torch.float64, device=d)
        self.j = torch.zeros_like(self.e)
        prof = w.ext_profile
        self.prof = None if prof is None else torch.from_numpy(prof).to(d)
        self.species = [self._locate(s) for s in w.species]

    def _hodge(self):
        """Galerkin edge mass matrix over the free edges: rows of up to five entries."""
        d = self.grad.device
        G = torch.einsum("fpk,fqk->fpq", self.grad, self.grad)
        I = (torch.ones(3, 3, dtype=torch.float64, device=d) + torch.eye(3, dtype=torch.float64, device=d)) * (self.area / 12.0)[:, None, None]
        loc = torch.zeros(self.nf, 3, 3, dtype=torch.float64, device=d)
        for m in range(3):
            a, b = (m + 1) % 3, (m + 2) % 3
            for n in range(3):
                c, e = (n + 1) % 3, (n + 2) % 3
                loc[:, m, n] = I[:, a, c] * G[:, b, e] - I[:, a, e] * G[:, b, c] - I[:, b, c] * G[:, a, e] + I[:, b, e] * G[:, a, c]
        loc = loc * self.ts[:, :, None] * self.ts[:, None, :]    # times eps0
        self.local_eps = loc
        idx = torch.full((self.ne,), -1, dtype=torch.long, device=d)
        idx[self.free] = torch.arange(len(self.free), device=d)
        row = idx[self.te][:, :, None].expand(-1, 3, 3).reshape(-1)
        col = idx[self.te][:, None, :].expand(-1, 3, 3).reshape(-1)
        ok = (row >= 0) & (col >= 0)
        n = len(self.free)
        A = torch.sparse_coo_tensor(torch.stack([row[ok], col[ok]]), loc.reshape(-1)[ok], (n, n)).coalesce()
        r, c = A.indices()
        start = torch.searchsorted(r, torch.arange(n, device=d))
        k = torch.arange(len(r), device=d) - start[r]
        self.a_col = torch.full((n, 5), -1, dtype=torch.long, device=d)
        self.a_val = torch.zeros(n, 5, dtype=torch.float64, device=d)
        self.a_col[r, k], self.a_val[r, k] = c, A.values()

    def _inverse(self):
        """Level-2 sparse approximate inverse: per column the least-squares solution on its neighbours'
        neighbours, by the normal equations; then symmetrised."""
        d, n, W = self.a_col.device, len(self.a_col), 13
        big = n
        ac, av = torch.cat([self.a_col, torch.full((1, 5), -1, device=d)]), torch.cat([self.a_val, torch.zeros(1, 5, dtype=torch.float64, device=d)])
        cand = ac[torch.where(self.a_col >= 0, self.a_col, big)].reshape(n, 25)
        cand = torch.where(cand >= 0, cand, big).sort(1).values
        cand[:, 1:] = torch.where(cand[:, 1:] == cand[:, :-1], big, cand[:, 1:])
        J = cand.sort(1).values[:, :W].contiguous()
        V = torch.zeros(n, W, dtype=torch.float64, device=d)
        for lo in range(0, n, 20000):
            Jc = J[lo:lo + 20000]
            kc, kv = ac[Jc], av[Jc]                              # [c, W, 5]
            G = torch.zeros(len(Jc), W, W, dtype=torch.float64, device=d)
            for s in range(5):
                for t in range(5):
                    same = (kc[:, :, None, s] == kc[:, None, :, t]) & (kc[:, :, None, s] >= 0)
                    G += torch.where(same, kv[:, :, None, s] * kv[:, None, :, t], 0.0)
            me = torch.arange(lo, lo + len(Jc), device=d)
            rhs = torch.where(kc == me[:, None, None], kv, 0.0).sum(2)
            G += torch.diag_embed((Jc == big).double())
            L = torch.linalg.cholesky(G)
            V[lo:lo + len(Jc)] = torch.cholesky_solve(rhs[:, :, None], L)[:, :, 0]
        V = torch.where(J == big, 0.0, V)
        Jp, Vp = torch.cat([J, torch.full((1, W), -1, device=d)]), torch.cat([V, torch.zeros(1, W, dtype=torch.float64, device=d)])
        for lo in range(0, n, 50000):
            Jc = J[lo:lo + 50000]
            me = torch.arange(lo, lo + len(Jc), device=d)
            back = torch.where(Jp[Jc] == me[:, None, None], Vp[Jc], 0.0).sum(2)
            V[lo:lo + len(Jc)] = 0.5 * (Vp[lo:lo + len(Jc)] + back)
        V = torch.where(J == big, 0.0, V) / EPS0
        self.m_col, self.m_val = self.free[J.clamp(max=n - 1)], V

    def _lam(self, f, r):
        return (self.grad[f] * (r[:, None, :] - self.far[f])).sum(2)

    def _locate(self, s):
        x, u = torch.from_numpy(s.x).cuda(), torch.from_numpy(s.u).cuda()
        hint = torch.from_numpy(s.hint).cuda().long()
        f = hint.clamp(min=0)
        bad = torch.nonzero((hint < 0) | (self._lam(f, x) < 0).any(1)).reshape(-1)
        every = torch.arange(self.nf, device=x.device)
        for k in bad.tolist():
            f[k] = torch.nonzero((self._lam(every, x[k].expand(self.nf, 2)) >= 0).all(1))[0, 0]
        return dict(q=float(s.q), m=float(s.m), x=x, u=u.clone(), f=f)

    @staticmethod
    def _push(pusher, u, E, B, alpha):
        def gam(v):
            return torch.sqrt(1.0 + (v * v).sum(1) / (C * C))

        def turn(v, t):
            """v + v x (t z)"""
            return torch.stack([v[:, 0] + v[:, 1] * t, v[:, 1] - v[:, 0] * t], 1)

        eps, be = alpha * E, alpha * B
        bb = be * be
        if pusher == "vay":
            v = u / gam(u)[:, None]
            un = u + 2.0 * eps + torch.stack([v[:, 1] * be, -v[:, 0] * be], 1)
            sig = gam(un) ** 2 - bb
            g = torch.sqrt(0.5 * (sig + torch.sqrt(sig * sig + 4.0 * bb)))
            t = be / g
            return turn(un, t) / (1.0 + t * t)[:, None], g
        um = u + eps
        g = gam(um)
        if pusher == "hc":
            sig = g * g - bb
            t = be / torch.sqrt(0.5 * (sig + torch.sqrt(sig * sig + 4.0 * bb)))
        elif pusher == "boris_tan":
            t = torch.tan(be / g)
        else:
            t = be / g
        up = turn(um, t)
        out = um + torch.stack([up[:, 1], -up[:, 0]], 1) * (2.0 * t / (1.0 + t * t))[:, None] + eps
        return out, gam(out)

    def step(self, pusher, amplitude=1.0):
        w, dt = self.w, self.dt
        se = self.e[self.te] * self.ts
        old = self.b
        self.b = old - dt * se.sum(1)
        bz = (self.b + old) * self.inv2a
        cur = torch.zeros(self.ne, dtype=torch.float64, device=se.device)
        for s in self.species:
            f, x = s["f"], s["x"]
            lam, g = self._lam(f, x), self.grad[f]
            E = torch.zeros_like(x)
            for m in range(3):
                a, b = (m + 1) % 3, (m + 2) % 3
                E += se[f, m][:, None] * (lam[:, a, None] * g[:, b] - lam[:, b, None] * g[:, a])
            we, wb = (1.0, 1.0) if self.prof is None else (self.prof[f, 0][:, None], self.prof[f, 1])
            E = E + amplitude * we * torch.tensor(w.ext[:2], dtype=torch.float64, device=x.device)
            s["u"], gam = self._push(pusher, s["u"], E, bz[f] + wb * w.ext[2], s["q"] * dt / (2.0 * s["m"]))
            end = x + s["u"] / gam[:, None] * dt
            self._walk(s, lam, end, cur)
        self.j = cur
        # Ampere: e += dt M (C^T [*mu^-1] b - i)
        h = torch.zeros_like(cur)
        h.index_add_(0, self.te.reshape(-1), (self.ts * (self.b / (MU0 * self.area))[:, None]).reshape(-1))
        r = h - cur
        self.e[self.free] += dt * (self.m_val * r[self.m_col]).sum(1)

    def _walk(self, s, lam, end, cur):
        """Split each path r(t) = start + t (end - start) per crossed triangle; deposit every piece."""
        scale = s["q"] / self.dt
        u = s["u"]
        idx = torch.arange(len(end), device=end.device)
        f, lo, hi, at, entry = s["f"].clone(), s["x"], end, torch.zeros_like(end[:, 0]), torch.full_like(idx, -1)
        out_f, out_x = s["f"], end.clone()
        for _ in range(64):
            l0, l1 = self._lam(f, lo), self._lam(f, hi)
            den = l0 - l1
            t = torch.maximum(torch.where(den > 0, l0 / torch.where(den > 0, den, 1.0), at[:, None]), at[:, None])
            no = (l1 >= 0) | (torch.arange(3, device=f.device)[None] == entry[:, None])
            t = torch.where(no, math.inf, t)
            tb, k = t.min(1)
            leaves = torch.isfinite(tb)
            lout = torch.where(leaves[:, None], l0 + torch.where(leaves, tb, 0.0)[:, None] * (l1 - l0), l1)
            lout = torch.where(leaves[:, None] & (torch.arange(3, device=f.device)[None] == k[:, None]), 0.0, lout)
            for m in range(3):
                a, b = (m + 1) % 3, (m + 2) % 3
                cur.index_add_(0, self.te[f, m], self.ts[f, m] * scale * (lam[:, a] * lout[:, b] - lout[:, a] * lam[:, b]))
            out_f[idx] = f
            out_x[idx] = hi
            go = torch.nonzero(leaves).reshape(-1)
            if len(go) == 0:
                break
            idx, f, lo, hi, k, at, lout = idx[go], f[go], lo[go], hi[go], k[go], tb[go], lout[go]
            nb = self.nb[f, k]
            wall = nb < 0
            # a wall turns the rest of the path and the momentum about its normal
            g = self.grad[f, k]
            hit = lo + at[:, None] * (hi - lo)
            gg = (g * g).sum(1)
            turned = hi - 2.0 * (((hi - hit) * g).sum(1) / gg)[:, None] * g
            uu = u[idx]
            u[idx] = torch.where(wall[:, None], uu - 2.0 * ((uu * g).sum(1) / gg)[:, None] * g, uu)
            step = torch.zeros_like(hi)
            if self.period is not None:
                step = self.shift[f, k][:, None] * self.period
            m2 = torch.where(wall, 0, nb % 3)
            # the neighbour's node m2+1 is our node k+2, its m2+2 our k+1
            hand = torch.zeros_like(lout)
            hand.scatter_(1, ((m2 + 1) % 3)[:, None], lout.gather(1, ((k + 2) % 3)[:, None]))
            hand.scatter_(1, ((m2 + 2) % 3)[:, None], lout.gather(1, ((k + 1) % 3)[:, None]))
            lam = torch.where(wall[:, None], lout, hand)
            f = torch.where(wall, f, nb // 3)
            entry = torch.where(wall, k, m2)
            lo = torch.where(wall[:, None], hit, lo + step)
            hi = torch.where(wall[:, None], turned, hi + step)
            at = torch.where(wall, 0.0, at)
        s["x"], s["f"] = out_x, out_f

    def energy(self):
        """e.[*eps].e / 2 + b.[*mu^-1].b / 2"""
        et = self.e[self.te]
        ee = EPS0 * torch.einsum("fm,fmn,fn->", et, self.local_eps, et)
        return float(0.5 * ee + 0.5 * (self.b * self.b / (MU0 * self.area)).sum())

    def probe(self, xy):
        """E at points, from the edge unknowns."""
        p = torch.from_numpy(xy).cuda()
        every = torch.arange(self.nf, device=p.device)
        if not hasattr(self, "at"):
            self.at = torch.tensor([int(torch.nonzero((self._lam(every, q.expand(self.nf, 2)) >= 0).all(1))[0, 0]) for q in p],
                                   device=p.device)
        lam, g, se = self._lam(self.at, p), self.grad[self.at], self.e[self.te[self.at]] * self.ts[self.at]
        E = torch.zeros_like(p)
        for m in range(3):
            a, b = (m + 1) % 3, (m + 2) % 3
            E += se[:, m, None] * (lam[:, a, None] * g[:, b] - lam[:, b, None] * g[:, a])
        return E


def exact(case, seed):
    ws = _workloads(case, seed)
    sims = [_Plain(w) for w in ws]
    if case["kind"] == "rf":
        w, drive, rows, P = ws[0], inputs.RFDrive(ws[0].ext[2], ws[0].dt, True), [], sims[0]
        for _ in range(case["steps"]):
            P.step(case["pusher"], drive.amplitude())
            x, u = P.species[0]["x"], P.species[0]["u"]
            drive.advance(_np(u))
            rows.append(torch.cat([x[0], u[0]]))
        return {"orbit": torch.stack(rows), "e": P.e, "b": P.b, "j": P.j}
    probes, energy, check = [], [0.0] * len(sims), case.get("check", 0)
    for k in range(case["steps"]):
        for P in sims:
            P.step(case["pusher"])
        if check and (k + 1) % check == 0:
            energy = [P.energy() for P in sims]
        if case.get("probes"):
            probes.append(sims[0].probe(_probe_line(ws[0].mesh, case["probes"])))
    single = case["precision"] == "fp32"
    out = {n: torch.cat([s[n] for P in sims for s in P.species]) for n in ("x", "u")}
    if not single:
        out["cell"] = torch.cat([s["f"] for P in sims for s in P.species]).int()
    for n in ("e", "b", "j"):
        out[n] = torch.cat([getattr(P, n) for P in sims])
    if probes:
        out["probes"] = torch.stack(probes)
    if check:
        out["continuity"], out["gauss"], out["energy"] = True, True, energy
    return out
