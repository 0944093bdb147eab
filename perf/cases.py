"""Timed cases of the Generalized Born / constant-(pH,E) / replica-exchange path.

Each case is work that a program hands to the package: force evaluations and
Born radii of single molecules and of batches, the differentiable energy, MD
segments with Monte Carlo halts and exchanges, and per-residue sweeps.  The
molecules are compact self-avoiding chains (bonds of 1.5 A, no two atoms
within 1.2 A, 0.05 atoms per cubic Angstrom) with the radii, charges and site
kinds that the package's synthetic workloads use.
"""
import math

import numpy as np
import torch

import paper_1803_09652_gb300 as pkg

KT = pkg.KB * 300.0
RADII = (1.2, 1.5, 1.7, 1.8, 2.0)
SCREEN = 0.8
DENSITY, STEP, CLASH = 0.05, 1.5, 1.2
E0_REF, PKA_REF = -0.203, (4.4, 4.85)
DEVICE = "cuda:0"

# site mixes: number of (redox, protonatable) residues
SITES = {"none": (0, 0), "peptide": (1, 1), "heme": (1, 3), "grid": (8, 32)}


def listed():
    return [
        # one force call on the 237-atom peptide of the paper's benchmark, as an outside MD engine makes it
        # at every step: launches and latency
        {"name": "forces_1x237", "kind": "forces", "replicas": 1, "atoms": 237, "kappa": 0.0, "cutoff": 0.0},
        # constant-(pH,E) MD of one small peptide: ten steps, then both Monte Carlo attempts
        {"name": "md_1x256", "kind": "md", "replicas": 1, "atoms": 256, "sites": "peptide", "n_pH": 1, "steps": 10,
         "cutoff": 0.0},
        # a screen of many small ragged molecules (33 to 300 atoms) in one call
        {"name": "forces_ragged_40x33to300", "kind": "forces", "replicas": 40, "atoms": 300, "atoms_min": 33,
         "kappa": 0.0, "cutoff": 0.0},
        # redox-potential replica exchange: eight replicas on an E ladder, an exchange every ten steps (50 per ps)
        {"name": "md_eremd_8x2048", "kind": "md", "replicas": 8, "atoms": 2048, "sites": "heme", "n_pH": 1, "steps": 10,
         "cutoff": 0.0},
        # forces of odd-sized molecules in salt water (Debye length 8 A)
        {"name": "forces_salt_3x4999", "kind": "forces", "replicas": 3, "atoms": 4999, "kappa": 0.125, "cutoff": 0.0},
        # Born radii of a batch of structures (fixed-radius scoring, Monte Carlo on fixed structures)
        {"name": "born_16x4096", "kind": "born", "replicas": 16, "atoms": 4096},
        # energy and its gradient in positions and charges inside a torch program, forward and backward
        {"name": "autograd_1x10007", "kind": "autograd", "replicas": 1, "atoms": 10007},
        # every protonatable residue of four large molecules tried once at fixed radii
        {"name": "sweep_4x25000", "kind": "sweep", "replicas": 4, "atoms": 25000, "sites": "grid"},
        # MD of a batch of unlike molecules, 500 to 20,000 atoms, with Monte Carlo halts
        {"name": "md_uneven_24x500to20000", "kind": "md", "replicas": 24, "atoms": 20000, "atoms_min": 500,
         "sites": "heme", "n_pH": 1, "steps": 10, "cutoff": 0.0},
        # forces of one large assembly with both cutoffs at 12 A
        {"name": "forces_cutoff_1x100000", "kind": "forces", "replicas": 1, "atoms": 100000, "kappa": 0.0,
         "cutoff": 12.0},
        # the two-dimensional (pH, E) exchange grid of 25,000-atom molecules: the largest batch (a few steps a
        # call, since the trajectories of crowded chains this size part from rounding alone within ten)
        {"name": "md_grid_48x25000", "kind": "md", "replicas": 48, "atoms": 25000, "sites": "grid", "n_pH": 6,
         "steps": 4, "cutoff": 0.0},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["forces", "forces", "md", "md", "born", "autograd", "sweep"])
    if kind == "sweep":
        return {"kind": kind, "replicas": rng.randint(1, 6), "atoms": _log(rng, 1000, 25000), "sites": "grid"}
    if kind == "autograd":
        return {"kind": kind, "replicas": rng.randint(1, 4), "atoms": _log(rng, 40, 10000)}
    if kind == "born":
        return {"kind": kind, "replicas": _log(rng, 1, 16), "atoms": _log(rng, 40, 10000)}
    replicas = _log(rng, 1, 24)
    atoms = _log(rng, 200, 20000 if replicas < 6 else 6000)
    if kind == "forces":
        c = {"kind": kind, "replicas": replicas, "atoms": atoms, "kappa": rng.choice([0.0, 0.0, 0.125]),
             "cutoff": rng.choice([0.0, 0.0, 0.0, 12.0, 16.0])}
    else:
        c = {"kind": kind, "replicas": replicas, "atoms": atoms, "sites": rng.choice(["peptide", "heme"]), "n_pH": 1,
             "steps": 10 if atoms <= 6000 else 4, "cutoff": 0.0}
    if rng.random() < 0.3 and replicas > 1:
        c["atoms_min"] = max(100, atoms // rng.choice([2, 8]))
    return c


# --- molecules -------------------------------------------------------------------

def _chain(n, rng):
    """A self-avoiding walk in the sphere that holds n atoms at the density: float32 [n, 3]."""
    side = 1 << 10
    offs = [(a * side + b) * side + c for a in (-1, 0, 1) for b in (-1, 0, 1) for c in (-1, 0, 1)]
    r2_max = (3.0 * n / (4.0 * math.pi * DENSITY)) ** (2.0 / 3.0)
    c2, inv, half = CLASH * CLASH, 1.0 / CLASH, side // 2
    pos, keys, grid = [(0.0, 0.0, 0.0)], [], {}
    key = (half * side + half) * side + half
    keys.append(key)
    grid[key] = [pos[0]]
    pool, at, fails = [], 0, 0
    while len(pos) < n:
        x, y, z = pos[-1]
        placed = False
        for _ in range(60):
            if at == len(pool):
                d = rng.normal(size=(8192, 3))
                pool, at = (d * (STEP / np.linalg.norm(d, axis=1, keepdims=True))).tolist(), 0
            dx, dy, dz = pool[at]
            at += 1
            px, py, pz = x + dx, y + dy, z + dz
            if px * px + py * py + pz * pz > r2_max:
                continue
            k = ((int(px * inv + half) * side) + int(py * inv + half)) * side + int(pz * inv + half)
            free = True
            for o in offs:
                for qx, qy, qz in grid.get(k + o, ()):
                    if (px - qx) ** 2 + (py - qy) ** 2 + (pz - qz) ** 2 < c2:
                        free = False
                        break
                if not free:
                    break
            if free:
                p = (px, py, pz)
                pos.append(p)
                keys.append(k)
                grid.setdefault(k, []).append(p)
                placed = True
                break
        if placed:
            fails = max(0, fails - 1)
        else:                              # a dead end: back up, further the more often it fails
            fails += 4
            for _ in range(min(fails, len(pos) - 1)):
                grid[keys.pop()].remove(pos.pop())
    return np.asarray(pos, np.float32)


def _molecule(n, sites, rng):
    """(xyzq [n, 4], rad_screen [n, 2], site list of (kind, first atom, charges per state))."""
    xyzq = np.zeros((n, 4), np.float32)
    xyzq[:, :3] = _chain(n, rng)
    q = rng.normal(0.0, 0.3, n)
    xyzq[:, 3] = q - q.mean()
    rad = np.full((n, 2), SCREEN, np.float32)
    rad[:, 0] = np.asarray(RADII, np.float32)[rng.integers(0, len(RADII), n)]
    redox, proton = SITES[sites]
    count, found = redox + proton, []
    for s in range(count):
        kind = 1 if s < redox else 0
        room = n // count
        size = min(int(rng.integers(8, 31)), room)
        first = s * room + int(rng.integers(0, room - size + 1))
        states = 2 if kind else int(rng.integers(2, 5))
        qs = np.repeat(xyzq[None, first:first + size, 3], states, 0).astype(np.float64)
        dq = rng.normal(0.0, 0.1, (states - 1, size))
        qs[1:] += dq + (1.0 - dq.sum(1, keepdims=True)) / size
        found.append((kind, first, qs.astype(np.float32)))
    return xyzq, rad, found


def _reference_energies(x, qs):
    """Energy of each charge set of a lone residue with all radii 3 A: its reference compound."""
    r2 = ((x[:, None] - x[None]) ** 2).sum(-1)
    f = np.sqrt(r2 + 9.0 * np.exp(-r2 / 36.0))
    np.fill_diagonal(r2, np.inf)
    a = pkg.KE * (1.0 / np.sqrt(r2) - (1.0 - 1.0 / 78.5) / f)
    return 0.5 * np.einsum("ka,ab,kb->k", qs, a, qs)


def _batch(case, seed):
    """Atom offsets, xyzq and rad_screen of the batch and its site table (the layout SiteTables takes)."""
    rng = np.random.default_rng([seed, 11])
    m, n, low = case["replicas"], case["atoms"], case.get("atoms_min")
    sites = case.get("sites", "none")
    if low:                                # unlike molecules, sizes spread over their logarithm
        sizes = [int(round(math.exp(v))) for v in rng.permutation(np.linspace(math.log(low), math.log(n), m))]
        mols = [_molecule(k, sites, rng) for k in sizes]
    else:                                  # copies of one molecule, as replica exchange starts
        mols = [_molecule(n, sites, rng)] * m
    off = np.concatenate([[0], np.cumsum([len(v[0]) for v in mols])]).astype(np.int64)
    t = {k: [0] for k in ("site_off", "site_atom_off", "site_state_off", "site_q_off")}
    t.update({k: [] for k in ("site_kind", "site_nstates", "site_atom_idx", "q_state", "G_ref", "n_H", "n_e",
                              "pKa_ref", "E0_ref")})
    for xyzq, _, found in mols:
        for kind, first, qs in found:
            states, size = qs.shape
            t["site_kind"].append(kind)
            t["site_nstates"].append(states)
            t["site_atom_idx"].extend(range(first, first + size))
            t["site_atom_off"].append(t["site_atom_off"][-1] + size)
            t["site_state_off"].append(t["site_state_off"][-1] + states)
            t["site_q_off"].append(t["site_q_off"][-1] + qs.size)
            t["q_state"].extend(qs.reshape(-1).tolist())
            t["G_ref"].extend(_reference_energies(xyzq[first:first + size, :3].astype(np.float64),
                                                  qs.astype(np.float64)).tolist())
            t["n_H"].extend([0] * states if kind else [0] + [1] * (states - 1))
            t["n_e"].extend([1, 0] if kind else [0] * states)
            t["pKa_ref"].append(0.0 if kind else PKA_REF[first % 2])
            t["E0_ref"].append(E0_REF if kind else 0.0)
        t["site_off"].append(len(t["site_kind"]))
    kinds = {"q_state": np.float32, "G_ref": np.float64, "pKa_ref": np.float64, "E0_ref": np.float64}
    table = {k: np.asarray(v, kinds.get(k, np.int32)) for k, v in t.items()}
    table["n_sites"] = len(t["site_kind"])
    return off, np.concatenate([v[0] for v in mols]), np.concatenate([v[1] for v in mols]), table


def _params(case):
    return dict(kappa=case.get("kappa", 0.0), rgbmax=case.get("cutoff", 0.0), cut=case.get("cutoff", 0.0))


def _fixed_radii(rad, seed):
    """Radii of an earlier evaluation, as a sweep is given them: the spread of compact chains."""
    rng = np.random.default_rng([seed, 12])
    return (rad[:, 0] * np.exp(rng.uniform(0.3, 2.8, len(rad)))).astype(np.float32)


def prepare(case, seed):
    off, xyzq, rad, table = _batch(case, seed)
    kind = case["kind"]
    if kind == "md":
        m, n_pH = case["replicas"], case["n_pH"]
        n_E = m // n_pH
        E_lad = E0_REF - 0.2 + 0.4 * np.arange(n_E) / max(n_E - 1, 1)
        pH_lad = 3.5 + 0.5 * np.arange(n_pH) if n_pH > 1 else np.full(1, 4.85)
        ladder = {} if case.get("atoms_min") else {"E_ladder": E_lad, "pH_ladder": pH_lad}   # copies exchange
        sim = pkg.Simulation(off, xyzq, rad, pkg.default_params(rep_k=100.0, rep_sigma=2.5, **_params(case)),
                             sites=table, pH=np.repeat(pH_lad, n_E), E=np.tile(E_lad, n_pH), **ladder, seed=seed,
                             mc_every=case["steps"], ex_every=case["steps"])
        return {"kind": kind, "sim": sim, "steps": case["steps"]}
    state = {"kind": kind, "ctx": pkg.Context(off, pkg.default_params(**_params(case))),
             "xyzq": torch.as_tensor(xyzq, device=DEVICE), "rad": torch.as_tensor(rad, device=DEVICE)}
    if kind == "autograd":
        state["xyzq"].requires_grad_(True)
    if kind == "sweep":
        m = case["replicas"]
        state["R"] = torch.as_tensor(_fixed_radii(rad, seed), device=DEVICE)
        state["sites"] = pkg.SiteTables(table, m, DEVICE)
        state["state"] = torch.zeros(table["n_sites"], dtype=torch.int32, device=DEVICE)
        state["pH"] = torch.full((m,), 4.85, dtype=torch.float64, device=DEVICE)
        state["E"] = torch.full((m,), E0_REF, dtype=torch.float64, device=DEVICE)
        state["seed"] = seed
    return state


def run(state):
    kind = state["kind"]
    if kind == "md":
        sim = state["sim"].run(state["steps"])
        return {"xyzq": sim.xyzq, "vel": sim.vel, "force": sim.force, "R": sim.R, "state": sim.state,
                "grid": sim.grid, "E": sim.E, "pH": sim.pH}
    ctx, xyzq, rad = state["ctx"], state["xyzq"], state["rad"]
    if kind == "born":
        return {"R": ctx.born_radii(xyzq, rad)}
    if kind == "forces":
        return ctx.energy_forces(xyzq, rad, want=("R", "F"))
    if kind == "autograd":
        # the pair terms are FP32: the program keeps energies in the type of its other tensors
        energy = pkg.GBEnergy.apply(ctx, xyzq, rad).float()
        grad, = torch.autograd.grad(energy.sum(), xyzq)
        return {"E": energy.detach(), "grad": grad}
    dG, acc = ctx.mc_sweep(state["sites"], xyzq, state["R"], state["pH"], state["E"], KT, state["seed"], 10, 0,
                           state["state"])
    return {"dG": dG, "acc": acc, "state": state["state"], "xyzq": xyzq}


def _sizes(case):
    m, n, low = case["replicas"], case["atoms"], case.get("atoms_min")
    if not low:
        return [n] * m
    return [int(round(math.exp(v))) for v in np.linspace(math.log(low), math.log(n), m)]


def work(case):
    """Far-field arithmetic of every pair that counts (fused multiply-add = 2), arrays read and written once."""
    sizes, kind = _sizes(case), case["kind"]
    n = sum(sizes)
    cut = case.get("cutoff", 0.0)
    near = DENSITY * 4.0 / 3.0 * math.pi * cut ** 3
    pairs = sum(k * (min(k - 1, near) if cut else k - 1) / 2 for k in sizes)
    if kind == "born":
        return {"bytes": 24 * n + 4 * n, "flops": 24 * pairs}
    if kind == "sweep":
        atoms = SITES[case["sites"]][1] * min(19, min(sizes) // sum(SITES[case["sites"]]))
        return {"bytes": 20 * n + 4 * n, "flops": 20 * atoms * n}
    if kind == "md":
        return {"bytes": case["steps"] * (16 + 16 + 16 + 8 + 16 + 16 + 16 + 4) * n,
                "flops": case["steps"] * 100 * pairs}
    return {"bytes": 24 * n + 16 * n, "flops": 100 * pairs}


# --- the same outputs in 64 bits ---------------------------------------------------

def _pairs(x, reach):
    """Ordered pairs i != j of one molecule (within reach, if there is one), a chunk at a time."""
    n = len(x)
    rows = max(1, (60_000_000 if reach else 3_000_000) // n)
    cols = torch.arange(n, device=x.device)
    for a in range(0, n, rows):
        i = torch.arange(a, min(n, a + rows), device=x.device)
        keep = i[:, None] != cols[None]
        if reach:
            keep &= torch.cdist(x[i], x, compute_mode="donot_use_mm_for_euclid_dist") < reach
        at, j = torch.nonzero(keep, as_tuple=True)
        yield i[at], j


def _hct(r, a, s, rc):
    """The pairwise descreening integral, over the ball of radius rc if there is one."""
    up = torch.clamp(r + s, max=rc) if rc else r + s
    low = torch.maximum(a, (r - s).abs())
    h = 1 / low - 1 / up + (r - s * s / r) / 4 * (1 / up ** 2 - 1 / low ** 2) + torch.log(low / up) / (2 * r)
    h = torch.where(low < up, h, torch.zeros_like(h))
    if rc:
        low = torch.clamp(low, max=rc)
    return 0.5 * (h + torch.where(a < s - r, 2 * (1 / a - 1 / low), torch.zeros_like(h)))


def _molecule64(xyzq, rad, case):
    """R, E_GB + E_Coulomb, dE/dx and dE/dq of one molecule."""
    p = {k: float(v) for k, v in _params(case).items()}
    f32 = lambda v: float(np.float32(v))  # noqa: E731  (the parameters are held in float32)
    kappa, rc, cut = f32(p["kappa"]), f32(p["rgbmax"]), f32(p["cut"])
    x, q = xyzq[:, :3].double().clone().requires_grad_(True), xyzq[:, 3].double().clone().requires_grad_(True)
    rho, n = rad[:, 0].double(), len(xyzq)
    a = rho - f32(0.09)
    s = rad[:, 1].double() * a
    kc, ko = pkg.KE, pkg.KE / 78.5
    integral = torch.zeros(n, dtype=torch.float64, device=x.device)
    with torch.no_grad():
        for i, j in _pairs(x, rc and rc + 2.0):
            integral.index_add_(0, i, _hct((x[i] - x[j]).norm(dim=1), a[i], s[j], rc))
    integral.requires_grad_(True)
    psi = a * integral
    R = 1 / (1 / a - torch.tanh(f32(1.0) * psi - f32(0.8) * psi ** 2 + f32(4.85) * psi ** 3) / rho)
    Rf = R.detach().clone().requires_grad_(True)
    screen = lambda f: kc - ko * torch.exp(-kappa * f)  # noqa: E731
    self_e = -0.5 * (screen(Rf) * q * q / Rf).sum()
    self_e.backward()
    energy = self_e.detach()
    for i, j in _pairs(x.detach(), cut):
        r2 = ((x[i] - x[j]) ** 2).sum(1)
        rr = Rf[i] * Rf[j]
        f = torch.sqrt(r2 + rr * torch.exp(-r2 / (4 * rr)))
        e = 0.5 * (q[i] * q[j] * (kc / torch.sqrt(r2) - screen(f) / f)).sum()
        e.backward()
        energy = energy + e.detach()
    c, = torch.autograd.grad(R, integral, Rf.grad)
    for i, j in _pairs(x.detach(), rc and rc + 2.0):
        (c[i] * _hct((x[i] - x[j]).norm(dim=1), a[i], s[j], rc)).sum().backward()
    return R.detach(), energy, x.grad, q.grad


def _philox(c, k):
    """Philox4x64-10 (Salmon et al., SC'11) on Python integers."""
    mask = (1 << 64) - 1
    c, k = list(c), list(k)
    for _ in range(10):
        p0, p1 = 0xD2E7470EE14C6C93 * c[0], 0xCA5A826395121157 * c[2]
        c = [(p1 >> 64) ^ c[1] ^ k[0], p1 & mask, (p0 >> 64) ^ c[3] ^ k[1], p0 & mask]
        k = [(k[0] + 0x9E3779B97F4A7C15) & mask, (k[1] + 0xBB67AE8584CAA73B) & mask]
    return c


def _sweep64(case, seed):
    """The sweep of mc_sweep: sites in random order, each tried with the charges left by those before it."""
    off, xyzq, rad, t = _batch(case, seed)
    x = torch.as_tensor(xyzq[:, :3], device=DEVICE).double()
    R = torch.as_tensor(_fixed_radii(rad, seed), device=DEVICE).double()
    charges = xyzq[:, 3].astype(np.float64)
    dG, acc, states = np.zeros(t["n_sites"]), np.full(t["n_sites"], 2, np.uint8), np.zeros(t["n_sites"], np.int32)
    tau = pkg.KE * (1.0 - 1.0 / 78.5)
    pick = lambda w, n: ((w >> 32) * n) >> 32  # noqa: E731
    for r in range(case["replicas"]):
        lo, hi = int(off[r]), int(off[r + 1])
        order = [s for s in range(t["site_off"][r], t["site_off"][r + 1]) if t["site_kind"][s] == 0]
        atoms = np.concatenate([t["site_atom_idx"][t["site_atom_off"][s]:t["site_atom_off"][s + 1]] for s in order])
        where = {s: np.searchsorted(atoms, t["site_atom_idx"][t["site_atom_off"][s]:t["site_atom_off"][s + 1]])
                 for s in order}
        ia = torch.as_tensor(atoms, device=DEVICE).long()
        xr, Rr = x[lo:hi], R[lo:hi]
        r2 = ((xr[ia][:, None] - xr[None]) ** 2).sum(-1)
        rr = Rr[ia][:, None] * Rr[None]
        A = pkg.KE / torch.sqrt(r2) - tau / torch.sqrt(r2 + rr * torch.exp(-r2 / (4 * rr)))
        A[torch.arange(len(ia)), ia] = -tau / Rr[ia]
        phi = (A @ torch.as_tensor(charges[lo:hi], device=DEVICE)).cpu().numpy()
        A = A[:, ia].cpu().numpy()
        for v in range(len(order)):
            w = _philox((r, 10, 5, v), (seed, 0))
            k = v + pick(w[0], len(order) - v)
            order[v], order[k] = order[k], order[v]
            s = order[v]
            at, size = where[s], len(where[s])
            new = pick(w[1], int(t["site_nstates"][s]) - 1)
            new += new >= states[s]
            qo = t["site_q_off"][s] + new * size
            q_new = t["q_state"][qo:qo + size].astype(np.float64)
            g = lo + atoms[at]
            dq = q_new - charges[g]
            so = t["site_state_off"][s]
            dG[s] = dq @ phi[at] + 0.5 * dq @ A[np.ix_(at, at)] @ dq - (t["G_ref"][so + new] - t["G_ref"][so + states[s]])
            dG[s] += KT * math.log(10.0) * (4.85 - t["pKa_ref"][s]) * (t["n_H"][so + new] - t["n_H"][so + states[s]])
            acc[s] = dG[s] <= 0 or (w[2] >> 11) / 2.0 ** 53 < math.exp(-dG[s] / KT)
            if acc[s]:
                phi += A[:, at] @ dq
                charges[g], states[s] = q_new, new
    out = np.concatenate([xyzq[:, :3].astype(np.float64), charges[:, None]], 1)
    return {"dG": dG, "acc": acc, "state": states, "xyzq": out}


def exact(case, seed):
    kind = case["kind"]
    if kind == "md":                       # a trajectory: no 64-bit value of its own
        return None
    if kind == "sweep":
        return _sweep64(case, seed)
    off, xyzq, rad, _ = _batch(case, seed)
    xyzq, rad = torch.as_tensor(xyzq, device=DEVICE), torch.as_tensor(rad, device=DEVICE)
    same = not case.get("atoms_min")       # copies of one molecule
    per = [_molecule64(xyzq[off[r]:off[r + 1]], rad[off[r]:off[r + 1]], case)
           for r in range(1 if same else case["replicas"])]
    per = per * case["replicas"] if same else per
    R = torch.cat([v[0] for v in per])
    dx, dq = torch.cat([v[2] for v in per]), torch.cat([v[3] for v in per])
    if kind == "born":
        return {"R": R}
    if kind == "forces":
        return {"R": R, "F": -dx}
    return {"E": torch.stack([v[1] for v in per]), "grad": torch.cat([dx, dq[:, None]], 1)}
