"""The calls that users of the library make, with sizes, inputs and 64-bit results, for measurement.

A case is one call through the Python interface on one periodic system (or one
batch of systems): stochastic-Lanczos energies, energies with forces, a
molecular-dynamics step through autograd, products C x, the screening front
end, and a batch of boxes of uneven sizes.

A system in mixed precision evaluates the operator in 32 bits and returns its
numbers in 64-bit containers; the cases keep such results as the 32-bit numbers
that they are, as a program that stores them would.  Results of FP64 systems
stay 64 bits wide.
"""
from __future__ import annotations

import math

import numpy as np
import torch

WATER_DENSITY = 0.0049535       # molecules per bohr^3: liquid water at 1 g/cm^3
ATOM_DENSITY = 3 * WATER_DENSITY
ANGSTROM = 1.8897261254578281   # bohr
DAMP_BETA, DAMP_D = 0.83, 6.0
SCREEN_FREQ = 23                # quadrature nodes of the screening, and its tolerance
SCREEN_TOL = 1e-10


# ---------------------------------------------------------------------------- the cases
def _case(name, op, kind, atoms, mesh, probes=0, steps=0, precision="mixed", order=6, edge=0.0, skew=False,
          ewald_beta=0.30, r_cut=12.0):
    return {"name": name, "op": op, "kind": kind, "atoms": atoms, "edge": edge, "skew": skew, "mesh": mesh,
            "order": order, "ewald_beta": ewald_beta, "r_cut": r_cut, "precision": precision, "probes": probes,
            "steps": steps}


def listed():
    return [
        # the smallest workload in full precision: a unit cell of 64 atoms, where launches and waits count
        _case("forces_64_fp64", "forces", "random", 64, "32x32x32", 16, 30, "fp64", edge=24.0, ewald_beta=0.35,
              r_cut=10.0),
        # the mesh-convergence box of 96 molecules at the density of points that the method suggests: one probe
        _case("energy_288_one_probe", "energy", "water", 288, "27x27x27", 1, 30, "fp64"),
        # one product C x, as an iterative eigensolver asks for: a crystal cell of 512 atoms
        _case("apply_512_one_vector", "apply", "diamond", 512, "27x27x27", 1),
        # an odd request: skew cell, odd atom and probe counts, a mesh of three lengths, spline order 8
        _case("energy_1371_skew_order8", "energy", "random", 1371, "45x48x50", 33, 24, order=8, edge=45.2,
              skew=True, ewald_beta=0.35, r_cut=10.0),
        # a block of products C x on a box of 1000 molecules
        _case("apply_3000_block", "apply", "water", 3000, "64x64x64", 64),
        # the everyday run: energy and forces of 1000 molecules
        _case("forces_3000", "forces", "water", 3000, "64x64x64", 64, 50),
        # its check in full precision
        _case("energy_3000_fp64", "energy", "water", 3000, "64x64x64", 32, 30, "fp64"),
        # screening of the polarisabilities ahead of a run
        _case("screen_12000", "screen", "water", 12000, "96x96x96"),
        # many boxes of uneven sizes at once
        {"name": "batch_16", "op": "batch", "members": 16, "atoms": 200, "atoms_max": 6000, "precision": "mixed",
         "probes": 32, "steps": 40},
        # a molecular-dynamics step: new positions, energy, gradient
        _case("md_12000", "md", "water", 12000, "96x96x96", 64, 60),
        # larger boxes, up to the largest that the method is quoted on
        _case("forces_24000", "forces", "water", 24000, "128x128x128", 128, 60),
        _case("forces_100002", "forces", "water", 100002, "192x192x192", 64, 60),
    ]


def _smooth(n):
    """The smallest product of 2, 3 and 5 that is at least n."""
    k = max(1, math.ceil(n - 1e-9))
    while True:
        m = k
        for f in (2, 3, 5):
            while m % f == 0:
                m //= f
        if m == 1:
            return k
        k += 1


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["forces", "forces", "energy", "energy", "apply", "apply", "md", "screen", "batch"])
    if op == "batch":
        return {"op": "batch", "members": rng.randint(3, 24), "atoms": _log_int(rng, 100, 400),
                "atoms_max": _log_int(rng, 800, 6000), "precision": "mixed", "probes": rng.randint(8, 48),
                "steps": rng.randint(15, 45)}
    precision = "fp64" if rng.random() < 0.25 else "mixed"
    kind = rng.choice(["water", "water", "random"])
    atoms = _log_int(rng, 64, 3000 if precision == "fp64" else 24000)
    if kind == "water":
        atoms = 3 * max(24, atoms // 3)
    probes, steps = _log_int(rng, 1, 128), rng.randint(10, 60)
    if precision == "fp64":
        while atoms * probes * steps > 3000 * 32 * 30 and probes > 1:
            probes = (probes + 1) // 2
    edge = max(24.0, (atoms / ATOM_DENSITY) ** (1.0 / 3.0)) if kind == "random" else 0.0
    box = edge or (atoms / ATOM_DENSITY) ** (1.0 / 3.0)
    order = rng.choice([6, 6, 6, 4, 8])
    mesh = "x".join(str(_smooth(max(2 * order, box / rng.uniform(0.85, 1.1)))) for _ in range(3))
    r_cut = round(min(rng.uniform(9.0, 12.0), 0.46 * box), 2)
    case = {"op": op, "kind": kind, "atoms": atoms, "edge": edge, "skew": kind == "random" and rng.random() < 0.4,
            "mesh": mesh, "order": order, "ewald_beta": round(3.6 / r_cut, 3), "r_cut": r_cut, "precision": precision,
            "probes": probes, "steps": steps}
    if op == "apply":
        case["steps"] = 0
    if op == "screen":
        case["steps"] = case["probes"] = 0
    return case


# ---------------------------------------------------------------------------- inputs
class _Box:
    """A periodic system: cell, positions and per-atom parameters."""

    def __init__(self, cell, pos, alpha, omega, r_vdw, mesh, order, ewald_beta, r_cut):
        self.cell, self.pos, self.alpha, self.omega, self.r_vdw = cell, pos, alpha, omega, r_vdw
        self.mesh, self.spline_order, self.ewald_beta = mesh, order, ewald_beta
        self.r_cut = self.damp_cut = r_cut
        self.damp_beta, self.damp_d = DAMP_BETA, DAMP_D


def _lattice_points(rng, n, sides):
    """n sites of a sides[0] x sides[1] x sides[2] lattice, in order."""
    grid = np.stack(np.meshgrid(*[np.arange(k) for k in sides], indexing="ij"), -1).reshape(-1, 3)
    if len(grid) > n:
        grid = grid[np.sort(rng.permutation(len(grid))[:n])]
    return grid


def _water(rng, n_mol):
    """Rigid molecules on a jittered lattice with random orientations; molecules with an atom closer than 2.5 bohr
    to a neighbour's are turned again (up to a few close ones that stay)."""
    box = (n_mol / WATER_DENSITY) ** (1.0 / 3.0)
    side = math.ceil(n_mol ** (1.0 / 3.0) - 1e-9)
    grid = _lattice_points(rng, n_mol, (side,) * 3)
    oxygen = (grid + 0.5) * (box / side) + rng.uniform(-0.5, 0.5, (n_mol, 3))
    half = math.radians(104.5) / 2
    local = 1.81 * np.array([[0, 0, 0], [math.sin(half), 0, math.cos(half)], [-math.sin(half), 0, math.cos(half)]])

    def turned(at):
        q = rng.normal(size=(len(at), 4))
        w, x, y, z = (q / np.linalg.norm(q, axis=1, keepdims=True)).T
        rot = np.array([[1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w)],
                        [2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w)],
                        [2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)]])
        return oxygen[at, None, :] + np.einsum("ijm,aj->mai", rot, local)

    site = np.full((side,) * 3, -1)
    site[tuple(grid.T)] = np.arange(n_mol)
    offsets = [o for o in np.ndindex(3, 3, 3) if o > (1, 1, 1)]
    near = [site[tuple(((grid + np.array(o) - 1) % side).T)] for o in offsets]
    pos = turned(np.arange(n_mol))
    close = np.arange(n_mol)
    for _ in range(40):
        check = np.zeros(n_mol, bool)
        check[close] = True
        bad = []
        for other in near:
            a = np.nonzero((other >= 0) & (check | check[other]))[0]
            d = pos[a][:, :, None, :] - pos[other[a]][:, None, :, :]
            d -= box * np.round(d / box)
            bad.append(a[(np.sum(d * d, -1) < 2.5 ** 2).any((1, 2))])
        close = np.unique(np.concatenate(bad))
        if not len(close):
            break
        pos[close] = turned(close)
    oxy = np.tile([True, False, False], n_mol)
    return (np.eye(3) * box, np.mod(pos.reshape(-1, 3), box),
            np.where(oxy, 5.4, 2.5) * rng.uniform(0.9, 1.1, 3 * n_mol), np.where(oxy, 0.45, 0.55),
            np.where(oxy, 3.2, 3.1))


def _random(rng, n, edge, skew):
    """Atoms on a jittered lattice, at least 2.5 bohr apart at the density of water's atoms."""
    cell = np.eye(3) * edge
    if skew:
        cell = edge * np.array([[1.0, 0.0, 0.0], [0.12, 1.0, 0.0], [-0.08, 0.15, 1.0]])
    side = math.ceil(n ** (1.0 / 3.0) - 1e-9)
    pos = ((_lattice_points(rng, n, (side,) * 3) + 0.5) / side) @ cell
    pos += rng.uniform(-0.5, 0.5, (n, 3)) * max(0.0, min(1.5, edge / side - 2.5))
    return cell, pos, rng.uniform(5, 15, n), rng.uniform(0.3, 0.6, n), rng.uniform(3, 4, n)


def _diamond(rng, n):
    """Conventional cubic cells of diamond with thermal displacements."""
    side = round((n / 8) ** (1.0 / 3.0))
    frac = np.array([[0, 0, 0], [0, .5, .5], [.5, 0, .5], [.5, .5, 0]])
    frac = np.concatenate([frac, frac + 0.25])
    cells = np.stack(np.meshgrid(*[np.arange(side)] * 3, indexing="ij"), -1).reshape(-1, 1, 3)
    a = 3.567 * ANGSTROM
    pos = (cells + frac).reshape(-1, 3) * a + rng.normal(scale=0.08, size=(n, 3))
    return (np.eye(3) * side * a, np.mod(pos, side * a), np.full(n, 12.0), np.full(n, 4 * 46.6 / (3 * 12.0 ** 2)),
            np.full(n, 3.59))


def _box(case, seed):
    rng = np.random.default_rng([1000, seed])
    mesh = tuple(int(k) for k in case["mesh"].split("x"))
    if case["kind"] == "water":
        parts = _water(rng, case["atoms"] // 3)
    elif case["kind"] == "diamond":
        parts = _diamond(rng, case["atoms"])
    else:
        parts = _random(rng, case["atoms"], case["edge"], case["skew"])
    return _Box(*parts, mesh, case["order"], case["ewald_beta"], case["r_cut"])


def _batch(case, seed):
    """Boxes of atom counts spread over the logarithm from atoms to atoms_max."""
    rng = np.random.default_rng([1004, seed])
    members = case["members"]
    sizes = np.exp(np.linspace(math.log(case["atoms"]), math.log(case["atoms_max"]), members)).round().astype(int)
    out = []
    for k, n in enumerate(sizes):
        edge = (n / ATOM_DENSITY) ** (1.0 / 3.0)
        out.append(_Box(*_random(rng, int(n), edge, False), (_smooth(max(12, edge)),) * 3, 6, 0.35,
                        min(10.0, 0.49 * edge)))
    return out


def _probe_seed(seed):
    return 2307022780 + 7919 * (seed % 1000003)


def _vectors(case, seed):
    gen = torch.Generator().manual_seed(seed % (1 << 31))
    return torch.randn((case["probes"], 3 * case["atoms"]), generator=gen, dtype=torch.float64)


def prepare(case, seed):
    import paper_2307_02278_gb300 as mbd

    if case["op"] == "batch":
        boxes = _batch(case, seed)
        seeds = np.array([_probe_seed(seed) + k for k in range(len(boxes))], dtype=np.uint64)
        return {"case": case, "batch": mbd.MBDBatch(boxes, precision=case["precision"]), "seeds": seeds}
    box = _box(case, seed)
    state = {"case": case, "system": mbd.MBDSystem.from_workload(box, precision=case["precision"]),
             "seed": _probe_seed(seed)}
    if case["op"] == "apply":
        state["x"] = _vectors(case, seed).cuda()
    if case["op"] == "md":
        state["pos"] = torch.tensor(box.pos, dtype=torch.float64, device="cuda", requires_grad=True)
        state["mbd_energy"] = mbd.mbd_energy
    return state


# ---------------------------------------------------------------------------- the calls
def _kept(case, x):
    """The numbers that a program keeps: 32 bits wide from a mixed system."""
    if case["precision"] == "fp64" or isinstance(x, float):
        return x
    return x.astype(np.float32) if isinstance(x, np.ndarray) else x.float()


def run(state):
    case = state["case"]
    op, r, m = case["op"], case["probes"], case.get("steps", 0)
    if op == "batch":
        energies, traces = state["batch"].lanczos_energy(r, m, state["seeds"])
        return {"energies": _kept(case, energies), "traces": _kept(case, traces)}
    s = state["system"]
    if op == "forces":
        energy, forces = s.energy_forces(r, m, state["seed"])
        return {"energy": energy, "forces": _kept(case, forces)}
    if op == "energy":
        energy, more = s.lanczos_energy(r, m, state["seed"], details=True)
        return {"energy": energy, "trace": more["trace"], "q": _kept(case, more["q"])}
    if op == "apply":
        return {"y": _kept(case, s.apply_C(state["x"]))}
    if op == "md":
        energy = state["mbd_energy"](state["pos"], s, r, m, state["seed"])
        (gradient,) = torch.autograd.grad(energy, state["pos"])
        return {"energy": _kept(case, energy.detach()), "gradient": _kept(case, gradient)}
    out = s.scs_screen(SCREEN_FREQ, SCREEN_TOL)
    return {k: _kept(case, out[k]) for k in ("alpha", "omega", "r_vdw", "c6", "alpha_iu")}


def _pairs_per_atom(atoms, volume, r_cut):
    return min(atoms, atoms / volume * 4.0 / 3.0 * math.pi * r_cut ** 3)


def _work(op, atoms, volume, r_cut, points, order, probes, steps):
    """Bytes: positions, parameters, vectors in and results out.  Operations of the method: a product C x takes two
    real transforms, spreading and gathering over order^3 points, the pairs, and the updates of the recurrence."""
    product = (5 * points * math.log2(points) + 12 * order ** 3 * atoms
               + 18 * atoms * _pairs_per_atom(atoms, volume, r_cut) + 40 * atoms)
    if op == "apply":
        return {"bytes": 8 * 7 * atoms + 2 * 8 * 3 * atoms * probes, "flops": probes * product}
    if op == "screen":
        pair = 60 + 18 * 3   # the tensor, and its product with three directions
        return {"bytes": 8 * 7 * atoms + 8 * atoms * (SCREEN_FREQ + 5),
                "flops": 20 * (SCREEN_FREQ + 1) * atoms * _pairs_per_atom(atoms, volume, r_cut) * pair}
    flops = probes * steps * (product + 30 * atoms)
    if op in ("forces", "md"):
        flops += 2 * probes * (product + steps * 3 * atoms)
    return {"bytes": 8 * 10 * atoms + 8 * probes, "flops": flops}


def work(case):
    if case["op"] == "batch":
        total = {"bytes": 0.0, "flops": 0.0}
        for n in np.exp(np.linspace(math.log(case["atoms"]), math.log(case["atoms_max"]), case["members"])):
            edge = (n / ATOM_DENSITY) ** (1.0 / 3.0)
            one = _work("energy", n, edge ** 3, min(10.0, 0.49 * edge), _smooth(max(12, edge)) ** 3, 6,
                        case["probes"], case["steps"])
            total = {k: total[k] + one[k] for k in total}
        return total
    points = math.prod(int(k) for k in case["mesh"].split("x"))
    volume = case["edge"] ** 3 or case["atoms"] / ATOM_DENSITY
    return _work(case["op"], case["atoms"], volume, case["r_cut"], points, case["order"], case["probes"],
                 case["steps"])


# ---------------------------------------------------------------------------- 64-bit results
def _spline(x, p):
    """The cardinal B-spline M_p at x, zero outside [0, p]."""
    if p == 1:
        return ((x >= 0) & (x < 1)).to(x.dtype)
    return (x * _spline(x, p - 1) + (p - x) * _spline(x - 1, p - 1)) / (p - 1)


def _block_csr(i, j, blocks, n, cols):
    """Sparse [n b, cols] matrix with the given [b, b] blocks at block rows i and block columns j."""
    b = blocks.shape[1]
    k = torch.arange(b, device=i.device)
    rows = (b * i[:, None, None] + k[:, None]).expand(-1, b, b).reshape(-1)
    columns = (b * j[:, None, None] + k).expand(-1, b, b).reshape(-1)
    order = torch.argsort(rows, stable=True)
    crow = torch.zeros(n * b + 1, dtype=torch.int64, device=i.device)
    crow[1:] = torch.cumsum(torch.bincount(rows, minlength=n * b), 0)
    return torch.sparse_csr_tensor(crow, columns[order], blocks.reshape(-1)[order], (n * b, cols))


class _Reference:
    """The smooth particle-mesh Ewald product C x, its gradient and its quadrature in 64 bits, in plain torch.
    Cells are wider than twice the cutoff, so that a pair has one image at most within it."""

    def __init__(self, box):
        self.box = box
        self.dev = dev = "cuda" if torch.cuda.is_available() else "cpu"
        t = lambda a: torch.tensor(np.asarray(a), dtype=torch.float64, device=dev)  # noqa: E731
        self.cell, self.pos, self.alpha, self.omega, self.r_vdw = (
            t(a) for a in (box.cell, box.pos, box.alpha, box.omega, box.r_vdw))
        self.n = len(self.pos)
        self.recip = torch.linalg.inv(self.cell).T          # rows a*_1, a*_2, a*_3
        self.volume = float(torch.linalg.det(self.cell))
        self.kdim = torch.tensor(box.mesh, device=dev)
        self.cmat = self.kdim[:, None] * self.recip         # du_beta / dR_alpha
        self.g = self.omega * torch.sqrt(self.alpha)
        self.pair_i, self.pair_j = self._find_pairs()

    def _pair_vectors(self, pos, i, j):
        d = pos[i] - pos[j]
        with torch.no_grad():
            shift = torch.round(d @ self.recip.T) @ self.cell
        return d - shift

    def _find_pairs(self):
        found = []
        chunk = max(1, 100_000_000 // self.n)
        for i0 in range(0, self.n, chunk):
            d = self.pos[i0:i0 + chunk, None, :] - self.pos[None, :, :]
            d -= torch.round(d @ self.recip.T) @ self.cell
            r2 = (d * d).sum(-1)
            i, j = torch.nonzero((r2 < self.box.r_cut ** 2) & (r2 > 0), as_tuple=True)
            found.append((i + i0, j))
        return torch.cat([f[0] for f in found]), torch.cat([f[1] for f in found])

    def _fermi(self, rho, i, j):
        rsum = self.r_vdw[i] + self.r_vdw[j]
        return 1 / (1 + torch.exp(-DAMP_D * (rho / (DAMP_BETA * rsum) - 1)))

    def _pair_tensors(self, pos, i, j):
        """The screened tensors less the damped part of the bare ones, [pairs, 3, 3]."""
        beta = self.box.ewald_beta
        d = self._pair_vectors(pos, i, j)
        r2 = (d * d).sum(-1)
        rho = torch.sqrt(r2)
        e = torch.exp(-beta ** 2 * r2) / math.sqrt(math.pi)
        b1 = (torch.erfc(beta * rho) / rho + 2 * beta * e) / r2
        b2 = (3 * b1 + 4 * beta ** 3 * e) / r2
        rest = 1 - self._fermi(rho, i, j)
        eye = torch.eye(3, dtype=d.dtype, device=d.device)
        diag, outer = b1 - rest / (rho * r2), b2 - 3 * rest / (rho * r2 * r2)
        return diag[:, None, None] * eye - outer[:, None, None] * d[:, :, None] * d[:, None, :]

    def _stencil(self, pos):
        """Mesh points [N, p^3] and gradients [N, p^3, 3] of the interpolation weights."""
        p, k = self.box.spline_order, self.kdim
        u = pos @ self.cmat.T
        base = torch.floor(u.detach())
        t = torch.arange(p, device=self.dev)
        x = (u - base)[:, :, None] + t
        m, dm = _spline(x, p), _spline(x, p - 1) - _spline(x - 1, p - 1)
        at = (base.long()[:, :, None] - t) % k[:, None]
        flat = (at[:, 0, :, None, None] * k[1] + at[:, 1, None, :, None]) * k[2] + at[:, 2, None, None, :]
        prod = lambda a, b, c: (a[:, 0, :, None, None] * b[:, 1, None, :, None]  # noqa: E731
                                * c[:, 2, None, None, :]).reshape(len(pos), -1)
        grad = torch.stack([prod(dm, m, m), prod(m, dm, m), prod(m, m, dm)], -1) @ self.cmat
        return flat.reshape(len(pos), -1), grad

    def build_operator(self):
        n, box = self.n, self.box
        points = math.prod(box.mesh)
        self.near = _block_csr(self.pair_i, self.pair_j, self._pair_tensors(self.pos, self.pair_i, self.pair_j), n,
                               3 * n)
        flat, grad = self._stencil(self.pos)
        s = flat.shape[1]
        self.gather = torch.sparse_csr_tensor(torch.arange(3 * n + 1, device=self.dev) * s,
                                              flat[:, None, :].expand(n, 3, s).reshape(-1),
                                              grad.transpose(1, 2).reshape(-1), (3 * n, points))
        order = torch.argsort(flat.reshape(-1), stable=True)
        crow = torch.zeros(points + 1, dtype=torch.int64, device=self.dev)
        crow[1:] = torch.cumsum(torch.bincount(flat.reshape(-1), minlength=points), 0) * 3
        columns = (3 * torch.div(order, s, rounding_mode="floor")[:, None]
                   + torch.arange(3, device=self.dev)).reshape(-1)
        self.spread = torch.sparse_csr_tensor(crow, columns, grad.reshape(-1, 3)[order].reshape(-1), (points, 3 * n))
        # influence function of the mesh, averaged over +-m on the Nyquist planes
        p, beta = box.spline_order, box.ewald_beta
        freq, moduli = [], []
        j = torch.arange(p - 1, device=self.dev, dtype=torch.float64)
        mj = _spline(j + 1, p)
        for k in box.mesh:
            m = torch.arange(k, device=self.dev, dtype=torch.float64)
            freq.append(torch.where(m <= k // 2, m, m - k))
            phase = 2 * math.pi * m[:, None] * j / k
            moduli.append(1 / ((torch.cos(phase) @ mj) ** 2 + (torch.sin(phase) @ mj) ** 2))
        vec = (freq[0][:, None, None, None] * self.recip[0] + freq[1][None, :, None, None] * self.recip[1]
               + freq[2][None, None, :, None] * self.recip[2])
        m2 = (vec * vec).sum(-1)
        b = moduli[0][:, None, None] * moduli[1][None, :, None] * moduli[2][None, None, :]
        g = b * torch.exp(-math.pi ** 2 * m2 / beta ** 2) / (math.pi * self.volume * m2)
        g[0, 0, 0] = 0
        minus = torch.roll(torch.flip(g, (0, 1, 2)), (1, 1, 1), (0, 1, 2))
        self.influence = (0.5 * (g + minus))[:, :, :box.mesh[2] // 2 + 1, None].contiguous()
        self.self_term = -4 * beta ** 3 / (3 * math.sqrt(math.pi))
        return self

    def potential(self, d):
        """phi on the mesh [points, R] of the dipoles d [3N, R]."""
        mesh = (self.spread @ d).reshape(*self.box.mesh, -1)
        spec = torch.fft.rfftn(mesh, dim=(0, 1, 2))
        spec *= self.influence
        phi = torch.fft.irfftn(spec, s=self.box.mesh, dim=(0, 1, 2), norm="forward")
        return phi.reshape(math.prod(self.box.mesh), -1)

    def field(self, d):
        return self.near @ d + self.gather @ self.potential(d) + self.self_term * d

    def product(self, x):
        g = self.g.repeat_interleave(3)[:, None]
        w2 = (self.omega ** 2).repeat_interleave(3)[:, None]
        return w2 * x + g * self.field(g * x)

    def probes(self, seed, count):
        """u = +-1 by the top bit of SplitMix64(seed + (l << 32) + i), normalised, [3N, count]."""
        dim = 3 * self.n
        with np.errstate(over="ignore"):
            z = (np.uint64(seed) + (np.arange(count, dtype=np.uint64) << np.uint64(32))[None, :]
                 + np.arange(dim, dtype=np.uint64)[:, None] + np.uint64(0x9E3779B97F4A7C15))
            z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
            z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        u = 1.0 - 2.0 * ((z ^ (z >> np.uint64(31))) >> np.uint64(63)).astype(np.float64)
        return torch.from_numpy(u / math.sqrt(dim)).to(self.dev)

    def quadrature(self, seed, count, steps, forces=False):
        """Energy, trace, q [count] and, for the forces, (v, C^-1/2 v)."""
        v = self.probes(seed, count)
        a, b, basis = [], [], []
        y, before, coupling = v, None, None
        for k in range(steps):
            if forces:
                basis.append(y)
            l = self.product(y)
            a.append((y * l).sum(0))
            if k + 1 < steps:
                l -= a[-1] * y
                if before is not None:
                    l -= coupling * before
                coupling = torch.linalg.norm(l, dim=0)
                b.append(coupling)
                before, y = y, l / coupling
        delta = torch.diag_embed(torch.stack(a, 1).cpu())
        if steps > 1:
            off = torch.diag_embed(torch.stack(b, 1).cpu(), 1)
            delta = delta + off + off.transpose(1, 2)
        theta, vec = torch.linalg.eigh(delta)
        q = (vec[:, 0, :] ** 2 * torch.sqrt(theta)).sum(1)
        trace = 3 * self.n / count * float(q.sum())
        energy = 0.5 * trace - 1.5 * float(self.omega.sum())
        if not forces:
            return energy, trace, q.numpy(), None
        c = (vec * (vec[:, 0, :] / torch.sqrt(theta))[:, None, :]).sum(2).to(self.dev)
        w = torch.zeros_like(v)
        for k in range(steps):
            w += c[:, k] * basis[k]
        return energy, trace, q.numpy(), (v, w)

    def gradient(self, v, w):
        """dE/dR = (1/4)(3N/R) sum_l (g w_l)^T (dT'/dR) (g v_l), [N, 3]."""
        g = self.g.repeat_interleave(3)[:, None]
        p, q = g * w, g * v
        n, r = self.n, v.shape[1]
        p3, q3 = p.reshape(n, 3, r), q.reshape(n, 3, r)
        total = torch.zeros((n, 3), dtype=torch.float64, device=self.dev)
        for i0 in range(0, len(self.pair_i), 200_000):
            i, j = self.pair_i[i0:i0 + 200_000], self.pair_j[i0:i0 + 200_000]
            weight = torch.bmm(p3[i], q3[j].transpose(1, 2))
            pos = self.pos.clone().requires_grad_(True)
            total += torch.autograd.grad((weight * self._pair_tensors(pos, i, j)).sum(), pos)[0]
        phi_p, phi_q = self.potential(p), self.potential(q)
        for i0 in range(0, n, 2000):
            pos = self.pos[i0:i0 + 2000].clone().requires_grad_(True)
            flat, grad = self._stencil(pos)
            weight = (torch.bmm(phi_q[flat], p3[i0:i0 + 2000].transpose(1, 2))
                      + torch.bmm(phi_p[flat], q3[i0:i0 + 2000].transpose(1, 2)))
            total[i0:i0 + 2000] += torch.autograd.grad((weight * grad).sum(), pos)[0]
        return 0.25 * 3 * n / r * total

    def screened(self):
        """The screening's results: conjugate gradients per frequency on the sparse dipole coupling."""
        t, w = np.polynomial.legendre.leggauss(SCREEN_FREQ)
        u = np.concatenate([[0.0], 0.5 * (1 + t) / (1 - t)])
        w = torch.tensor(w / (1 - t) ** 2, device=self.dev)
        i, j = self.pair_i, self.pair_j
        d = self._pair_vectors(self.pos, i, j)
        r2 = (d * d).sum(-1)
        rho = torch.sqrt(r2)
        rest = 1 - self._fermi(rho, i, j)
        eye = torch.eye(3, dtype=torch.float64, device=self.dev)
        unit = eye.repeat(self.n, 1)
        out = []
        for freq in u:
            a_u = self.alpha / (1 + (freq / self.omega) ** 2)
            s = (math.sqrt(2 / math.pi) * a_u / 3) ** (1 / 3)
            sigma = torch.sqrt(s[i] ** 2 + s[j] ** 2)
            x = rho / sigma
            far, e = torch.erf(x), 2 / math.sqrt(math.pi) * torch.exp(-x * x)
            diag = far / (r2 * rho) - e / (sigma * r2)
            outer = 3 * far / (r2 * r2 * rho) - 3 * e / (sigma * r2 * r2) - 2 * e / (sigma ** 3 * r2)
            blocks = rest[:, None, None] * (diag[:, None, None] * eye - outer[:, None, None] * d[:, :, None]
                                            * d[:, None, :])
            coupling = _block_csr(i, j, blocks, self.n, 3 * self.n)
            a3 = a_u.repeat_interleave(3)[:, None]
            sol = a3 * unit
            res = unit - sol / a3 - coupling @ sol
            z = a3 * res
            step = z
            rz = (res * z).sum(0)
            for _ in range(200):
                if float((res * res).sum(0).max()) <= 1e-26 * self.n:
                    break
                ap = step / a3 + coupling @ step
                f = rz / (step * ap).sum(0)
                sol = sol + f * step
                res = res - f * ap
                z = a3 * res
                new = (res * z).sum(0)
                step = z + new / rz * step
                rz = new
            out.append((sol * unit).sum(1).reshape(self.n, 3).mean(1))
        alpha_iu = torch.stack(out)
        c6 = 3 / math.pi * (w[:, None] * alpha_iu[1:] ** 2).sum(0)
        alpha = alpha_iu[0]
        return {"alpha": alpha, "omega": 4 * c6 / (3 * alpha ** 2), "r_vdw": self.r_vdw * (alpha / self.alpha) ** (1 / 3),
                "c6": c6, "alpha_iu": alpha_iu}


def exact(case, seed):
    op, r, m = case["op"], case["probes"], case.get("steps", 0)
    if op == "batch":
        done = [_Reference(b).build_operator().quadrature(_probe_seed(seed) + k, r, m)
                for k, b in enumerate(_batch(case, seed))]
        return {"energies": np.array([e[0] for e in done]), "traces": np.array([e[1] for e in done])}
    ref = _Reference(_box(case, seed))
    if op == "screen":
        return ref.screened()
    ref.build_operator()
    if op == "apply":
        return {"y": ref.product(_vectors(case, seed).to(ref.dev).T.contiguous()).T.contiguous()}
    if op == "energy":
        energy, trace, q, _ = ref.quadrature(_probe_seed(seed), r, m)
        return {"energy": energy, "trace": trace, "q": q}
    energy, _, _, (v, w) = ref.quadrature(_probe_seed(seed), r, m, forces=True)
    gradient = ref.gradient(v, w)
    if op == "md":
        return {"energy": torch.tensor(energy, dtype=torch.float64), "gradient": gradient}
    return {"energy": energy, "forces": -gradient}
