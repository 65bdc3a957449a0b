"""The work that users of this framework have it do, as cases that can be timed.

Every case goes through the package's public entry points: a trajectory chunk
of one system (`binding.MD`: steps, then the energies and a frame), a
single-point evaluation (`MD.set_state`, energy, virial, forces), a batch of
replicas (`binding.MDBatch`) and one step of a force-matching fit
(`autodiff.ForceMatch`).  Results of mixed-precision contexts are kept as
float32, the precision that the option asks for (and what trajectory files
store); those of FP64 contexts stay float64.
"""
import math

import numpy as np
import torch

from paper_2405_07898_gb300 import autodiff, binding
from paper_2405_07898_gb300 import inputs as I

KB_ACCEL = 9.648533215665e-3  # (eV/Angstrom/amu) -> Angstrom/fs^2
DT = 2.0                      # fs, the step of every workload
REBUILD = 10                  # steps between list builds (the default)
BCC_LIST, BCC_PAIRS, FCC_LIST, FCC_PAIRS = 26, 14, 54, 42


def listed():
    def md(name, cells, steps, precision="mixed", lattice="bcc", temperature=300.0, open_axes=0, alloy=False):
        return {"name": name, "kind": "md", "lattice": lattice, "nx": cells[0], "ny": cells[1], "nz": cells[2],
                "steps": steps, "precision": precision, "temperature": temperature, "open_axes": open_axes,
                "alloy": alloy}

    return [
        # an outer program drives a small system step by step (a thermostat, a
        # collective variable): one step, then energies, forces and state
        md("coupled_1024_mixed", (8, 8, 8), 1),
        # the 2,000-atom FP64 system that the trajectories are checked on
        md("chunk_2000_fp64", (10, 10, 10), 100, precision="fp64"),
        # trajectory chunks over the strong-scaling sweep at 1,000 K
        md("chunk_6750_mixed", (15, 15, 15), 100, temperature=1000.0),
        md("chunk_43904_mixed", (28, 28, 28), 100, temperature=1000.0),
        md("chunk_118638_mixed", (39, 39, 39), 100, temperature=1000.0),
        # the benchmark system, between two frames of its trajectory
        md("chunk_799496_mixed", (74, 74, 73), 100),
        # the same system by a user who wants FP64 throughout
        md("chunk_799496_fp64", (74, 74, 73), 10, precision="fp64"),
        # the copper-size free-surface slab: open axes, 42 interactions per atom
        md("slab_801792_mixed", (174, 192, 6), 100, lattice="fcc", temperature=290.0, open_axes=7),
        # a two-type alloy: the type-dependent tables
        md("alloy_184320_mixed", (48, 48, 40), 50, temperature=400.0, alloy=True),
        # single-point evaluation of configurations that arrive in host memory
        {"name": "static_314928_mixed", "kind": "static", "lattice": "bcc", "nx": 54, "ny": 54, "nz": 54,
         "precision": "mixed", "temperature": 1000.0},
        # the replica batch: 512 uneven systems, BCC and FCC, advanced together
        {"name": "batch_512_mixed", "kind": "batch", "replicas": 512, "n_min": 1024, "n_max": 16384, "steps": 50},
        # one gradient step of a force-matching fit over 64 configurations
        {"name": "fit_64x2000_fp64", "kind": "fit", "configs": 64, "nx": 10, "ny": 10, "nz": 10, "knots": 64},
    ]


def draw(rng):
    def cells(n_lo, n_hi, per_cell, least=5):
        n = math.exp(rng.uniform(math.log(n_lo), math.log(n_hi))) / per_cell
        edge = n ** (1.0 / 3.0)
        nx = max(least, round(edge * rng.uniform(0.7, 1.3)))
        ny = max(least, round(edge * rng.uniform(0.7, 1.3)))
        return nx, ny, max(least, min(round(n / (nx * ny)), int(800000 / (per_cell * nx * ny))))

    kind = rng.choice(["mixed"] * 5 + ["fp64"] * 2 + ["slab", "alloy", "static", "static", "batch", "fit"])
    if kind == "batch":
        n_min = rng.randrange(1024, 3000)
        return {"kind": "batch", "replicas": rng.randrange(24, 200), "n_min": n_min,
                "n_max": n_min + rng.randrange(500, 10000), "steps": rng.randrange(5, 40)}
    if kind == "fit":
        return {"kind": "fit", "configs": rng.randrange(8, 60), "nx": rng.randrange(5, 11), "ny": rng.randrange(6, 11),
                "nz": rng.randrange(6, 11), "knots": rng.randrange(24, 90)}
    temperature = float(rng.randrange(100, 1100))
    lattice = rng.choice(["bcc", "bcc", "fcc"])
    if kind == "static":
        nx, ny, nz = cells(1000, 400000, 2 if lattice == "bcc" else 4)
        return {"kind": "static", "lattice": lattice, "nx": nx, "ny": ny, "nz": nz,
                "precision": rng.choice(["mixed", "mixed", "fp64"]), "temperature": temperature}
    if kind == "alloy":
        lattice, temperature = "bcc", 400.0
    nx, ny, nz = cells(1000, {"mixed": 700000, "fp64": 100000, "slab": 700000, "alloy": 150000}[kind],
                       2 if lattice == "bcc" else 4)
    open_axes = 0
    if kind == "slab":
        open_axes = rng.randrange(1, 8)
        if open_axes & 4:  # thin along z
            nz, area = rng.randrange(3, 9), nx * ny * nz
            nx, ny = max(5, round(math.sqrt(area / nz) * 1.1)), max(5, round(math.sqrt(area / nz) / 1.1))
    atoms = nx * ny * nz * (2 if lattice == "bcc" else 4)
    longest = max(2, min(100, int(4e7 / atoms if kind != "fp64" else 2e6 / atoms)))
    return {"kind": "md", "lattice": lattice, "nx": nx, "ny": ny, "nz": nz,
            "steps": max(1, round(math.exp(rng.uniform(0.0, math.log(longest))))),
            "precision": "fp64" if kind == "fp64" else "mixed", "temperature": temperature, "open_axes": open_axes,
            "alloy": kind == "alloy"}


# --------------------------------------------------------------------------
# inputs


_potentials = {}


def _johnson(lattice):
    if lattice not in _potentials:
        _potentials[lattice] = I.johnson_potential(_params(lattice))
    return _potentials[lattice]


def _params(lattice):
    return I.BCC_TA_LIKE if lattice == "bcc" else I.FCC_CU_LIKE


def _system(case, seed):
    cells = (case["nx"], case["ny"], case["nz"])
    if case.get("alloy"):
        return I.multi_type_system(cells, seed=seed)
    p = _params(case["lattice"])
    pos, box = I.lattice(p, *cells)
    rng = np.random.Generator(np.random.PCG64(seed))
    pos += rng.normal(0.0, 0.02, size=pos.shape)
    box = box.copy()
    for a in range(3):
        if (case.get("open_axes", 0) >> a) & 1:  # a free surface with 6 Angstrom of vacuum
            pos[:, a] += 6.0
            box[a] += 12.0
        else:
            pos[:, a] = np.mod(pos[:, a], box[a])
    return I.System(box=box, pos=pos, vel=I.maxwell(pos.shape[0], p.mass, case["temperature"], rng),
                    types=np.zeros(pos.shape[0], np.int32), pot=_johnson(case["lattice"]),
                    open_axes=case.get("open_axes", 0))


def _replicas(case, seed):
    """Uneven systems, the first half BCC, the second FCC: sizes (near cubes of
    whole cells) and temperatures belong to the case, the states to the seed."""
    rng = np.random.Generator(np.random.PCG64(case["replicas"]))
    out = []
    for r in range(case["replicas"]):
        p = _params("bcc" if r < case["replicas"] // 2 else "fcc")
        atoms = math.exp(rng.uniform(math.log(case["n_min"]), math.log(case["n_max"])))
        cells, least = atoms / (2 if p.lattice == "bcc" else 4), math.ceil(3 * (p.r_cut + p.skin) / p.a)
        nx = max(least, round(cells ** (1 / 3)))
        ny = max(least, round(math.sqrt(cells / nx)))
        out.append(I.thermal_system(p, (nx, ny, max(least, round(cells / (nx * ny)))), 0.02,
                                    rng.uniform(200.0, 1200.0), 1000 * seed + r))
    return out


def _problem(case, seed):
    return I.fit_problem(case["configs"], (case["nx"], case["ny"], case["nz"]), case["knots"], seed=seed)


def _host(n, dtype=torch.float64):
    return torch.zeros((n, 3), dtype=dtype, pin_memory=torch.cuda.is_available())


def prepare(case, seed):
    state = {"case": case}
    if case["kind"] == "batch":
        systems = _replicas(case, seed)
        state["batch"] = binding.MDBatch(systems)
        state["sizes"] = [s.n for s in systems]
        n = sum(state["sizes"])
        state["out"] = {k: torch.zeros((n, 3), dtype=torch.float32) for k in ("pos", "vel", "force")}
        return state
    if case["kind"] == "fit":
        problem = _problem(case, seed)
        state["fit"] = autodiff.ForceMatch(problem)
        state["theta"] = problem.theta0.copy()
        return state
    system = _system(case, seed)
    n = system.n
    state["md"] = binding.MD(system, precision=case["precision"])
    state["host"] = {k: _host(n) for k in ("pos", "vel", "force")}
    if case["kind"] == "static":
        state["in_pos"], state["in_vel"] = _host(n), _host(n)
        state["in_pos"].copy_(torch.from_numpy(system.pos))
        state["in_vel"].copy_(torch.from_numpy(system.vel))
    if case["precision"] == "mixed":
        state["out"] = {k: torch.zeros((n, 3), dtype=torch.float32) for k in ("pos", "vel", "force")}
    return state


# --------------------------------------------------------------------------
# one pass


def _energies(case, *values):
    dtype = torch.float64 if case["precision"] == "fp64" else torch.float32
    return torch.tensor(values, dtype=dtype)


def _frame(state, keys):
    """The pass's arrays in the precision of the context."""
    if state["case"]["precision"] == "fp64":
        return {k: state["host"][k] for k in keys}
    return {k: state["out"][k].copy_(state["host"][k]) for k in keys}


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        b = state["batch"]
        b.step(case["steps"], DT)
        pe, ke = b.energy()
        at = 0
        for r, n in enumerate(state["sizes"]):
            for k, x in zip(("pos", "vel", "force"), b.get_state(r)):
                state["out"][k][at:at + n] = torch.from_numpy(x)
            at += n
        return {"pe": pe.astype(np.float32), "ke": ke.astype(np.float32), **state["out"]}
    if case["kind"] == "fit":
        loss, grad = state["fit"].evaluate(state["theta"], grad=True)
        state["theta"] = _descend(state["theta"], grad)
        return {"loss": np.array([loss]), "grad": grad, "theta": state["theta"]}
    md, host = state["md"], state["host"]
    if case["kind"] == "static":
        md.set_state(state["in_pos"], state["in_vel"])
        pe, ke = md.energy()
        virial = md.virial()
        md.forces(out=host["force"].numpy())
        return {"energy": _energies(case, pe, ke), "virial": _energies(case, *virial), **_frame(state, ("force",))}
    md.step(case["steps"], DT)
    pe, ke = md.energy()
    md.get_state(host["pos"], host["vel"])
    md.forces(out=host["force"].numpy())
    return {"energy": _energies(case, pe, ke), **_frame(state, ("pos", "vel", "force"))}


def _descend(theta, grad):
    """A short step along the gradient, relative to each knot's own size."""
    return theta - 1e-5 * (np.abs(theta) + 1e-3) * grad / (np.abs(grad) + 1e-2 * np.abs(grad).max())


# --------------------------------------------------------------------------
# what a pass cannot do without


def work(case):
    def per_atom(lattice):
        return (BCC_LIST, BCC_PAIRS) if lattice == "bcc" else (FCC_LIST, FCC_PAIRS)

    def steps_of(atoms, lattice, steps, wide):
        n_list, n_pair = per_atom(lattice)
        # a step: position and velocity in and out, each listed pair once;
        # a list build (every REBUILD steps): positions in, the list out
        byte = atoms * (steps * (4 * 24 + 2 * n_list) + steps / REBUILD * (24 + 2 * n_list))
        # a pair: distance, two spline lookups in the density and force sums
        return byte + atoms * 72 * (1 if wide else 0.5), atoms * steps * (n_pair / 2 * 70 + n_list / 2 * 10 + 40)

    if case["kind"] == "batch":
        mean = (case["n_max"] - case["n_min"]) / math.log(case["n_max"] / case["n_min"])
        half = [steps_of(case["replicas"] / 2 * mean, s, case["steps"], False) for s in ("bcc", "fcc")]
        return {"bytes": half[0][0] + half[1][0], "flops": half[0][1] + half[1][1]}
    if case["kind"] == "fit":
        atoms = case["configs"] * 2 * case["nx"] * case["ny"] * case["nz"]
        return {"bytes": atoms * (24 + 24 + 2 * BCC_LIST) + 6 * 8 * case["knots"], "flops": atoms * BCC_PAIRS / 2 * 300}
    atoms = case["nx"] * case["ny"] * case["nz"] * (2 if case["lattice"] == "bcc" else 4)
    if case["kind"] == "static":
        n_list, n_pair = per_atom(case["lattice"])
        return {"bytes": atoms * (48 + 24 + 2 * 2 * n_list), "flops": atoms * (n_pair / 2 * 70 + n_list / 2 * 10)}
    byte, flop = steps_of(atoms, case["lattice"], case["steps"], case["precision"] == "fp64")
    return {"bytes": byte, "flops": flop}


# --------------------------------------------------------------------------
# the same in 64 bits, in plain torch


def _spline(k):
    """Cubic spline through uniform knots from its second derivatives:
    rows (a, b, c, d) of S(t) = a + b t + c t^2 + d t^3 per interval."""
    return _spline_rows(torch.from_numpy(np.asarray(k.y, np.float64)), k).numpy()


def _spline_rows(y, k):
    """The rows as a (differentiable) function of the knot values y."""
    n, h = k.n, k.dx
    A = np.zeros((n, n))
    B = np.zeros((n, n))
    c = np.zeros(n)
    i = np.arange(1, n - 1)
    A[i, i - 1], A[i, i], A[i, i + 1] = h / 6, 2 * h / 3, h / 6
    B[i, i - 1], B[i, i], B[i, i + 1] = 1 / h, -2 / h, 1 / h
    A[0, 0] = A[n - 1, n - 1] = 1.0
    if k.bc_lo == 1:
        A[0, 0], A[0, 1], B[0, 0], B[0, 1], c[0] = h / 3, h / 6, -1 / h, 1 / h, -k.d_lo
    if k.bc_hi == 1:
        A[n - 1, n - 1], A[n - 1, n - 2], B[n - 1, n - 1], B[n - 1, n - 2], c[n - 1] = h / 3, h / 6, -1 / h, 1 / h, k.d_hi
    A, B, c = (torch.from_numpy(x).to(y.device) for x in (A, B, c))
    m = torch.linalg.solve(A, B @ y + c)
    return torch.stack([y[:-1], (y[1:] - y[:-1]) / h - h * (2 * m[:-1] + m[1:]) / 6, m[:-1] / 2,
                        (m[1:] - m[:-1]) / (6 * h)], 1)


class _Table:
    """Several splines with their own spacing, looked up by index."""

    def __init__(self, knots, device, rows=None):
        self.x0 = torch.tensor([k.x0 for k in knots], dtype=torch.float64, device=device)
        self.h = torch.tensor([k.dx for k in knots], dtype=torch.float64, device=device)
        self.n = torch.tensor([k.n - 1 for k in knots], device=device)
        rows = rows if rows is not None else [torch.from_numpy(_spline(k)).to(device) for k in knots]
        self.off = torch.tensor(np.cumsum([0] + [r.shape[0] for r in rows[:-1]]), device=device)
        self.rows = torch.cat(rows)

    def __call__(self, q, x, beyond=False):
        """Value and derivative of spline q at x; beyond: along the end
        tangents outside the knots."""
        h, x0 = self.h[q], self.x0[q]
        k = torch.minimum(torch.floor((x - x0) / h).long().clamp_(min=0), self.n[q] - 1)
        t = x - (x0 + k * h)
        over = torch.zeros_like(t)
        if beyond:
            inside = torch.minimum(t.clamp(min=0.0), h)
            over, t = t - inside, inside
        c = self.rows[self.off[q] + k]
        der = c[..., 1] + t * (2 * c[..., 2] + 3 * t * c[..., 3])
        return c[..., 0] + t * (c[..., 1] + t * (c[..., 2] + t * c[..., 3])) + over * der, der


class _Plain:
    """Atoms of one or many boxes under Eqs. 2-5 of the method, in FP64.
    Each atom has the box of its system; `group` separates the systems."""

    CHUNK = 1 << 15

    def __init__(self, pots, pot_of, sizes, boxes, pos, vel, types, open_axes=0):
        self.dev = dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
        reps = torch.tensor(sizes, device=dev)
        group = torch.repeat_interleave(torch.arange(len(sizes), device=dev), reps)
        lists = np.array([p.r_cut + p.skin for p in pots])
        grids = np.floor(np.array(boxes) / lists[np.array(pot_of), None]).astype(np.int64)
        first = np.concatenate([[0], np.cumsum(grids.prod(1))])
        self.ncells = int(first[-1])
        self.first = torch.from_numpy(first[:-1]).to(dev)[group]
        self.grid = torch.from_numpy(grids).to(dev)[group]
        self.box = torch.from_numpy(np.array(boxes, np.float64)).to(dev)[group]
        self.periodic = torch.tensor([not (open_axes >> a) & 1 for a in range(3)], device=dev)
        nt = [p.ntypes for p in pots]
        base = np.concatenate([[0], np.cumsum(nt)])[:-1]
        pair_base = np.concatenate([[0], np.cumsum([t * (t + 1) // 2 for t in nt])])[:-1]
        which = torch.tensor(pot_of, device=dev)[group]
        self.nt = torch.tensor(nt, device=dev)[which]
        self.own = torch.from_numpy(types.astype(np.int64)).to(dev)
        self.type = self.own + torch.from_numpy(base).to(dev)[which]
        self.pair_base = torch.from_numpy(pair_base).to(dev)[which]
        self.rc2 = torch.tensor([p.r_cut ** 2 for p in pots], dtype=torch.float64, device=dev)[which]
        self.rl2 = torch.from_numpy(lists ** 2).to(dev)[which]
        self.move2 = torch.tensor([0.25 * p.skin ** 2 for p in pots], dtype=torch.float64, device=dev)[which]
        self.mass = torch.tensor(np.concatenate([p.mass for p in pots]), dtype=torch.float64, device=dev)[self.type]
        self.F = _Table([k for p in pots for k in p.F], dev)
        self.f = _Table([k for p in pots for k in p.f], dev)
        self.phi = _Table([k for p in pots for k in p.phi], dev)
        self.group, self.ngroup = group, len(sizes)
        self.x = torch.from_numpy(np.ascontiguousarray(pos)).to(dev)
        self.v = torch.from_numpy(np.ascontiguousarray(vel)).to(dev)
        self.build()

    def build(self):
        dev, n = self.dev, self.x.shape[0]
        inside = (self.x >= 0) & (self.x < self.box)
        self.x = torch.where(inside | ~self.periodic, self.x, self.x - self.box * torch.floor(self.x / self.box))
        self.since = torch.zeros(self.ngroup, dtype=torch.int64, device=dev)
        self.ref = self.x.clone()
        c = torch.floor(self.x * (self.grid / self.box)).long()
        c = torch.maximum(torch.minimum(c, self.grid - 1), torch.zeros_like(c))
        cid = self.first + (c[:, 2] * self.grid[:, 1] + c[:, 1]) * self.grid[:, 0] + c[:, 0]
        order = torch.sort(cid, stable=True).indices
        start = torch.zeros(self.ncells + 1, dtype=torch.int64, device=dev)
        start[1:] = torch.cumsum(torch.bincount(cid, minlength=self.ncells), 0)
        most = torch.arange(int((start[1:] - start[:-1]).max()), device=dev)
        off = torch.tensor([[dx, dy, dz] for dz in (-1, 0, 1) for dy in (-1, 0, 1) for dx in (-1, 0, 1)], device=dev)
        rows, counts = [], []
        for a in range(0, n, self.CHUNK):
            i = torch.arange(a, min(n, a + self.CHUNK), device=dev)
            e = c[i][:, None, :] + off
            g = self.grid[i][:, None, :]
            there = ((e >= 0) & (e < g)) | self.periodic
            e = torch.remainder(e, g)
            e = self.first[i][:, None] + (e[..., 2] * g[..., 1] + e[..., 1]) * g[..., 0] + e[..., 0]
            s = start[e]
            cnt = torch.where(there.all(-1), start[e + 1] - s, torch.zeros_like(s))
            j = order[(s[..., None] + most).clamp_(max=n - 1)].view(len(i), -1)
            ok = (most < cnt[..., None]).view(len(i), -1) & (j != i[:, None])
            d = self.vector(i, j)
            ok &= (d * d).sum(-1) < self.rl2[i][:, None]
            counts.append(ok.sum(1))
            rows.append(j[ok])
        counts, rows = torch.cat(counts), torch.cat(rows)
        k = max(1, int(counts.max()))
        at = torch.arange(rows.numel(), device=dev) - torch.repeat_interleave(torch.cumsum(counts, 0) - counts, counts)
        self.j = torch.arange(n, device=dev)[:, None].repeat(1, k)
        self.j[torch.repeat_interleave(torch.arange(n, device=dev), counts), at] = rows
        self.listed = torch.arange(k, device=dev) < counts[:, None]

    def vector(self, i, j):
        d = self.x[j] - self.x[i][:, None, :]
        L = self.box[i][:, None, :]
        return d - torch.where(self.periodic, torch.round(d / L), torch.zeros_like(d)) * L

    def pairs(self, i):
        j = self.j[i]
        d = self.vector(i, j)
        r2 = (d * d).sum(-1)
        on = self.listed[i] & (r2 < self.rc2[i][:, None])
        r = torch.sqrt(torch.where(on, r2, torch.ones_like(r2)))
        lo, hi = torch.minimum(self.own[i][:, None], self.own[j]), torch.maximum(self.own[i][:, None], self.own[j])
        q = self.pair_base[i][:, None] + lo * self.nt[i][:, None] - lo * (lo - 1) // 2 + (hi - lo)
        return j, d, r, on.to(torch.float64), q

    def evaluate(self, virial=False):
        n = self.x.shape[0]
        chunks = [torch.arange(a, min(n, a + 4 * self.CHUNK), device=self.dev) for a in range(0, n, 4 * self.CHUNK)]
        rho = torch.empty(n, dtype=torch.float64, device=self.dev)
        for i in chunks:
            j, d, r, on, q = self.pairs(i)
            rho[i] = (self.f(self.type[j], r)[0] * on).sum(1)
        Fv, Fp = self.F(self.type, rho, beyond=True)
        self.force, pe, w = torch.empty_like(self.x), Fv, torch.zeros(6, dtype=torch.float64, device=self.dev)
        for i in chunks:
            j, d, r, on, q = self.pairs(i)
            ph, dph = self.phi(q, r)
            s = dph + Fp[i][:, None] * self.f(self.type[j], r)[1]
            s = (s + Fp[j] * self.f(self.type[i][:, None].expand_as(j), r)[1]) * on / r
            self.force[i] = (s[..., None] * d).sum(1)
            pe[i] += 0.5 * (ph * on).sum(1)
            if virial:
                w += torch.stack([-0.5 * (s * d[..., a] * d[..., b]).sum()
                                  for a, b in ((0, 0), (1, 1), (2, 2), (0, 1), (0, 2), (1, 2))])
        ke = (0.5 * self.mass / KB_ACCEL)[:, None] * self.v * self.v
        zero = torch.zeros(self.ngroup, dtype=torch.float64, device=self.dev)
        self.pe, self.ke = zero.index_add(0, self.group, pe), zero.index_add(0, self.group, ke.sum(1))
        return w

    def step(self, steps):
        self.evaluate()
        kick = (0.5 * DT * KB_ACCEL / self.mass)[:, None]
        moved = self.x.clone()  # as if no system were wrapped
        for _ in range(steps):
            self.v = self.v + kick * self.force
            self.x = self.x + DT * self.v
            self.since += 1
            far = ((self.x - self.ref).square().sum(1) > self.move2)
            far = torch.zeros(self.ngroup, device=self.dev).index_add(0, self.group, far.float()) > 0
            due = far | (self.since >= REBUILD)
            if bool(due.any()):
                # every list is built anew; only the systems that are due
                # wrap their positions and restart their count
                since, ref, x = self.since, self.ref, self.x
                self.build()
                here = due[self.group][:, None]
                self.since = torch.where(due, self.since, since)
                self.ref, self.x = torch.where(here, self.ref, ref), torch.where(here, self.x, x)
            self.evaluate()
            self.v = self.v + kick * self.force
        ke = (0.5 * self.mass / KB_ACCEL)[:, None] * self.v * self.v
        self.ke = torch.zeros(self.ngroup, dtype=torch.float64, device=self.dev).index_add(0, self.group, ke.sum(1))


def exact(case, seed):
    if case["kind"] == "fit":
        return _exact_fit(case, seed)
    if case["kind"] == "batch":
        systems = _replicas(case, seed)
        kinds = [0 if abs(s.pot.r_cut - I.BCC_TA_LIKE.r_cut) < 1e-9 else 1 for s in systems]
        plain = _Plain([_johnson("bcc"), _johnson("fcc")], kinds, [s.n for s in systems], [s.box for s in systems],
                       np.concatenate([s.pos for s in systems]), np.concatenate([s.vel for s in systems]),
                       np.concatenate([s.types for s in systems]))
        plain.step(case["steps"])
        return {"pe": plain.pe, "ke": plain.ke, "pos": plain.x, "vel": plain.v, "force": plain.force}
    s = _system(case, seed)
    plain = _Plain([s.pot], [0], [s.n], [s.box], s.pos, s.vel, s.types, s.open_axes)
    if case["kind"] == "static":
        virial = plain.evaluate(virial=True)
        return {"energy": torch.cat([plain.pe, plain.ke]), "virial": virial, "force": plain.force}
    plain.step(case["steps"])
    return {"energy": torch.cat([plain.pe, plain.ke]), "pos": plain.x, "vel": plain.v, "force": plain.force}


def _exact_fit(case, seed):
    p = _problem(case, seed)
    knots = I.johnson_knots(p.params, p.n_knots)  # F, f, phi: the grids and end conditions
    sizes, boxes = [c[0].shape[0] for c in p.configs], [c[1] for c in p.configs]
    pos = np.concatenate([c[0] for c in p.configs])
    plain = _Plain([_johnson("bcc")], [0] * len(sizes), sizes, boxes, pos, np.zeros_like(pos),
                   np.zeros(pos.shape[0], np.int64))
    plain.evaluate()
    e_ref, f_ref, dev, n = plain.pe, plain.force, plain.dev, p.n_knots
    theta = torch.from_numpy(p.theta0).to(dev).requires_grad_()
    parts = (theta[2 * n:], theta[n:2 * n], theta[:n])  # F, f, phi
    F, f, phi = (_Table([k], dev, [_spline_rows(y, k)]) for y, k in zip(parts, knots))
    every = torch.arange(pos.shape[0], device=dev)
    j, d, r, on, q = plain.pairs(every)
    zero = torch.zeros_like(q)
    fv, fd = f(zero, r)
    Fv, Fp = F(zero[:, 0], (fv * on).sum(1), beyond=True)
    ph, dph = phi(zero, r)
    force = (((dph + (Fp[:, None] + Fp[j]) * fd) * on / r)[..., None] * d).sum(1)
    e = torch.zeros(len(sizes), dtype=torch.float64, device=dev)
    e = e.index_add(0, plain.group, Fv + 0.5 * (ph * on).sum(1))
    count = torch.tensor(sizes, dtype=torch.float64, device=dev)
    loss = ((e - e_ref) ** 2 / count).sum() + p.w * ((force - f_ref) ** 2).sum()
    loss.backward()
    grad = theta.grad.cpu().numpy()
    return {"loss": np.array([loss.item()]), "grad": grad, "theta": _descend(p.theta0, grad)}
