"""Performance cases of the short-range nonbonded library and its PME mesh steps.

Each case is one pass of work that a molecular-dynamics program (or a
parameter fit) has the library do, through the package's public Python
entry points. Systems are rigid three-site water at liquid density, the
stand-in this repository uses everywhere: 33.4 molecules per nm^3, oxygens on
a jittered lattice, random orientations without close contacts, charges
-0.8476 / +0.4238 e, LJ on the oxygens, intramolecular exclusions. Inputs are
made on the GPU from the seed alone.

Kinds of case (``case["kind"]``):

``forces``   One evaluation between two prunes: forces (and, with ``energy``,
             energies) of the current frame over a pruned list whose prune is
             a few frames old. ``coul`` picks the Coulomb flavour.
``oneshot``  A single point: pair search and then forces and energies over
             the unpruned list.
``cycle``    One prune interval of a trajectory: search, prune, and the force
             calls of the frames that follow, forces only.
``adjoint``  A force-matching step: forces, their difference from the target
             forces (the gradient of half the squared error), and the loss's
             gradients with respect to positions, charges and the LJ matrix.
``batch``    Independent boxes of mixed sizes in one pair list: search,
             prune to the cutoff, forces and energies of every box.
``halo``     The local / non-local split of a domain decomposition: the local
             part, then the non-local part, on one stream.
``spread``   PME charge spreading onto the mesh (order 4).
``gather``   PME force gathering from a mesh potential (order 4).
"""
import math

import numpy as np
import torch

from paper_2405_01420_gb300 import nb

DEV = "cuda"
DENSITY = 33.4               # waters per nm^3
Q_O, Q_H = -0.8476, 0.4238   # e
SIGMA_O, EPS_O = 0.3166, 0.650
R_OH, THETA = 0.1, math.radians(109.47)
MIN_CONTACT = 0.15           # nm
COULOMB_F = 138.935458       # kJ mol^-1 nm e^-2
STEP = 0.001                 # nm, per frame and component, of a trajectory's random walk
F64 = torch.float64


def listed():
    return [
        # The smallest system in use, 512 waters, one MD step on a pruned list: latency and launches.
        {"name": "forces_1536", "kind": "forces", "waters": 512, "rc": 0.9, "rlist": 1.0, "r_inner": 0.95,
         "energy": False, "coul": "ewald"},
        # A single point on the same system: the first call of a program, or each call of one that keeps no list.
        {"name": "oneshot_1536", "kind": "oneshot", "waters": 512, "rc": 0.9},
        # An ordinary solvated peptide's size, an odd number of molecules and partly filled columns.
        {"name": "forces_11997", "kind": "forces", "waters": 3999, "rc": 1.0, "rlist": 1.1, "r_inner": 1.04,
         "energy": False, "coul": "ewald"},
        # The benchmark box with energies, as on the steps that write them.
        {"name": "forces_energy_96k", "kind": "forces", "waters": 32000, "rc": 1.0, "rlist": 1.1, "r_inner": 1.04,
         "energy": True, "coul": "ewald"},
        # The benchmark box over one prune interval: search, prune, ten force calls.
        {"name": "cycle_96k", "kind": "cycle", "waters": 32000, "rc": 1.0, "rlist": 1.1, "r_inner": 1.04,
         "frames": 10},
        # The largest system in use, one MD step.
        {"name": "forces_1m", "kind": "forces", "waters": 333334, "rc": 1.0, "rlist": 1.1, "r_inner": 1.04,
         "energy": False, "coul": "ewald"},
        # The reaction-field flavour with the excluded-pair correction, energies on, an odd size.
        {"name": "rf_energy_24k", "kind": "forces", "waters": 7999, "rc": 1.0, "rlist": 1.1, "r_inner": 1.04,
         "energy": True, "coul": "rf_excl"},
        # Force matching on the differentiation box: four LJ types, normal charges.
        {"name": "adjoint_24k", "kind": "adjoint", "waters": 8000, "rc": 1.0, "rlist": 1.1, "r_inner": 1.04},
        # The batched workload: 256 boxes of 1,536 to 24,000 atoms.
        {"name": "batch_256", "kind": "batch", "boxes": 256, "lo": 512, "hi": 8000, "rc": 0.9, "rlist": 1.0},
        # A domain with one neighbour: the atoms within the list radius of a face are halo atoms.
        {"name": "halo_96k", "kind": "halo", "waters": 32000, "rc": 1.0, "rlist": 1.1, "r_inner": 1.04},
        # The mesh steps on the benchmark box, mesh spacing at most 0.12 nm.
        {"name": "pme_spread_96k", "kind": "spread", "waters": 32000, "K": 84},
        {"name": "pme_gather_96k", "kind": "gather", "waters": 32000, "K": 84},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["forces", "forces", "forces", "oneshot", "cycle", "adjoint", "batch", "halo", "spread", "gather"])
    if kind == "batch":
        boxes = _log_int(rng, 3, 200)
        lo = rng.randint(300, 1500)
        return {"kind": kind, "boxes": boxes, "lo": lo, "hi": lo + rng.randint(100, 6000), "rc": 0.7, "rlist": 0.8}
    if kind in ("spread", "gather"):
        waters = _log_int(rng, 500, 300000)
        edge = (waters / DENSITY) ** (1.0 / 3.0)
        return {"kind": kind, "waters": waters, "K": _fft_size(int(math.ceil(edge / rng.choice([0.1, 0.12])))) + rng.choice([0, 0, 1])}
    if kind == "oneshot":
        return {"kind": kind, "waters": _log_int(rng, 400, 20000), "rc": rng.choice([0.8, 0.9])}
    rc = rng.choice([0.9, 1.0])
    case = {"kind": kind, "waters": 0, "rc": rc, "rlist": round(rc + 0.1, 3), "r_inner": round(rc + rng.choice([0.04, 0.05]), 3)}
    if kind == "forces":
        case["waters"] = _log_int(rng, 512, 300000)
        case["energy"] = rng.random() < 0.4
        case["coul"] = rng.choice(["ewald", "ewald", "ewald", "ewald_shift", "rf", "rf_excl"])
    elif kind == "cycle":
        case["waters"] = _log_int(rng, 512, 60000)
        case["frames"] = rng.randint(5, 10)
    elif kind == "adjoint":
        case["waters"] = _log_int(rng, 512, 20000)
    else:
        case["waters"] = _log_int(rng, 4000, 100000)
    return case


def _fft_size(n):
    while True:
        m = n
        for p in (2, 3, 5, 7):
            while m % p == 0:
                m //= p
        if m == 1:
            return n
        n += 1


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _rotations(k, gen):
    """k uniformly random rotation matrices (unit quaternions from normals)."""
    q = torch.randn((k, 4), generator=gen, device=DEV, dtype=F64)
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - z * w), 2 * (x * z + y * w),
                        2 * (x * y + z * w), 1 - 2 * (x * x + z * z), 2 * (y * z - x * w),
                        2 * (x * z - y * w), 2 * (y * z + x * w), 1 - 2 * (x * x + y * y)], dim=1).view(k, 3, 3)


def _water(sizes, gen):
    """Water boxes of the given numbers of molecules, back to back: positions
    [M, 3, 3] (FP64, unwrapped), the box edge of each molecule [M] and of
    each box. Molecules with an atom within 0.15 nm of a neighbour's get new
    orientations, up to 100 times."""
    edges = [(w / DENSITY) ** (1.0 / 3.0) for w in sizes]
    sides = []
    for w in sizes:
        n = int(round(w ** (1.0 / 3.0)))
        while n ** 3 < w:
            n += 1
        while (n - 1) ** 3 >= w and n > 1:
            n -= 1
        sides.append(n)
    sites, cell_off, mol_off = [], [], []
    cells = mols = 0
    for w, n in zip(sizes, sides):
        s = torch.randperm(n ** 3, generator=gen, device=DEV)[:w].sort().values if n ** 3 > w else torch.arange(w, device=DEV)
        sites.append(s)
        cell_off.append(cells)
        mol_off.append(mols)
        cells += n ** 3
        mols += w
    reps = torch.tensor(sizes, device=DEV)
    per = lambda v, t: torch.repeat_interleave(torch.tensor(v, dtype=t, device=DEV), reps)  # noqa: E731
    n, off, L = per(sides, torch.int64), per(cell_off, torch.int64), per(edges, F64)
    s = torch.cat(sites)
    sx, sy, sz = s // (n * n), (s // n) % n, s % n
    at = torch.full((cells,), -1, dtype=torch.int64, device=DEV)
    at[off + s] = torch.arange(mols, device=DEV)
    a = L / n
    oxy = (torch.stack([sx, sy, sz], dim=1) + 0.5) * a[:, None]
    oxy = oxy + (torch.rand((mols, 3), generator=gen, device=DEV, dtype=F64) * 2 - 1) * 0.05 * a[:, None]
    sn, cs = math.sin(THETA / 2), math.cos(THETA / 2)
    body = torch.tensor([[0.0, 0.0, 0.0], [R_OH * sn, 0.0, R_OH * cs], [-R_OH * sn, 0.0, R_OH * cs]], dtype=F64, device=DEV)
    pos = oxy[:, None, :] + torch.einsum("mij,aj->mai", _rotations(mols, gen), body)
    look = torch.arange(mols, device=DEV)  # molecules to look at
    for _ in range(100):
        bad = torch.zeros(mols, dtype=torch.bool, device=DEV)
        nn, Lm = n[look], L[look]
        for k in range(27):
            if k == 13:
                continue
            dx, dy, dz = k // 9 - 1, (k // 3) % 3 - 1, k % 3 - 1
            c = ((sx[look] + dx) % nn) * nn * nn + ((sy[look] + dy) % nn) * nn + (sz[look] + dz) % nn
            other = at[off[look] + c]
            ok = (other >= 0) & (other != look)
            d = pos[look][:, :, None, :] - pos[other.clamp(min=0)][:, None, :, :]
            d = d - Lm[:, None, None, None] * torch.round(d / Lm[:, None, None, None])
            bad[look] |= ok & ((d * d).sum(-1) < MIN_CONTACT ** 2).any(dim=2).any(dim=1)
        look = bad.nonzero()[:, 0]
        if look.numel() == 0:
            break
        pos[look] = oxy[look][:, None, :] + torch.einsum("mij,aj->mai", _rotations(look.numel(), gen), body)
    return pos, L, edges


def _wrapped(x, L):
    """FP64 positions [N, 3] in boxes of edge L [N] as FP32 in [0, L)."""
    L32 = L.float()[:, None]
    w = (x - L[:, None] * torch.floor(x / L[:, None])).float()
    return torch.where((w >= L32) | (w < 0), torch.zeros_like(w), w).contiguous()


def _exclusions(n):
    i = torch.arange(n, device=DEV)
    base, k = 3 * (i // 3), i % 3
    idx = torch.stack([base + (k + 1) % 3, base + (k + 2) % 3], dim=1).sort(dim=1).values
    return (2 * torch.arange(n + 1, device=DEV)).int().contiguous(), idx.reshape(-1).int().contiguous()


def _system(sizes, seed, halo=None):
    """A dict of what the calls take: positions, charges, types, LJ matrix,
    exclusions, box edges. With ``halo``, molecules whose oxygen lies within
    that distance of the upper x face come last."""
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    pos, L, edges = _water(sizes, gen)
    s = {}
    if halo is not None:
        ox = pos[:, 0, 0] - L * torch.floor(pos[:, 0, 0] / L)
        far = ox >= edges[0] - halo
        order = torch.cat([(~far).nonzero()[:, 0], far.nonzero()[:, 0]])
        pos = pos[order]
        s["n_home"] = 3 * int((~far).sum())
    n = 3 * pos.shape[0]
    s["n"] = n
    s["L"] = torch.repeat_interleave(L, 3)
    s["edges"] = edges
    s["x64"] = pos.reshape(n, 3)
    s["x"] = _wrapped(s["x64"], s["L"])
    s["box"] = [float(np.float32(edges[0]))] * 3
    s["q"] = torch.tensor([Q_O, Q_H, Q_H], dtype=torch.float32, device=DEV).repeat(n // 3)
    s["t"] = torch.tensor([0, 1, 1], dtype=torch.int32, device=DEV).repeat(n // 3)
    lj = np.zeros((2, 2, 2), dtype=np.float32)
    lj[0, 0] = 4 * EPS_O * SIGMA_O ** 6, 4 * EPS_O * SIGMA_O ** 12
    s["lj"] = torch.from_numpy(lj).to(DEV)
    s["eo"], s["ei"] = _exclusions(n)
    s["gen"] = gen
    return s


def _walk(s, frames):
    """The next frames of a random walk from the box's positions."""
    x, out = s["x64"], []
    for _ in range(frames):
        x = x + torch.randn(x.shape, generator=s["gen"], device=DEV, dtype=F64) * STEP
        out.append(_wrapped(x, s["L"]))
    return out


def _beta(rc):
    """Ewald splitting parameter with erfc(beta rc) = 1e-5."""
    lo, hi = 0.0, 10.0
    for _ in range(100):
        mid = 0.5 * (lo + hi)
        lo, hi = (mid, hi) if math.erfc(mid * rc) > 1e-5 else (lo, mid)
    return 0.5 * (lo + hi)


def _sizes(case, seed):
    if case["kind"] != "batch":
        return [case["waters"]]
    # the sizes of the boxes belong to the case: every seed has the same ones
    return [int(v) for v in np.random.default_rng(case["boxes"]).integers(case["lo"], case["hi"] + 1, case["boxes"])]


def _inputs(case, seed):
    """The case's inputs, without the library."""
    kind = case["kind"]
    s = _system(_sizes(case, seed), seed, halo=case["rlist"] if kind == "halo" else None)
    gen = s["gen"]
    if kind in ("forces", "halo"):
        s["frame"] = _walk(s, 4)[-1]
    elif kind == "cycle":
        s["frames"] = [s["x"]] + _walk(s, case["frames"] - 1)
    elif kind == "adjoint":
        n = s["n"]
        q = torch.randn(n, generator=gen, device=DEV, dtype=F64) * 0.4
        s["q"] = (q - q.mean()).float()
        s["t"] = torch.randint(0, 4, (n,), generator=gen, device=DEV).int()
        c6 = 1e-3 + 2e-3 * torch.rand(4, generator=gen, device=DEV, dtype=F64)
        c12 = 1e-6 + 2e-6 * torch.rand(4, generator=gen, device=DEV, dtype=F64)
        s["lj"] = torch.stack([torch.outer(c6, c6).sqrt(), torch.outer(c12, c12).sqrt()], dim=-1).float().contiguous()
        s["target_noise"] = torch.randn((n, 3), generator=gen, device=DEV, dtype=F64)
        s["frame"] = _walk(s, 4)[-1]
    elif kind == "gather":
        # a mesh potential as the solve leaves it: normal charges through the reciprocal-space kernel
        K, L = case["K"], s["edges"][0]
        rho = torch.randn((K, K, K), generator=gen, device=DEV, dtype=F64)
        m = torch.fft.fftfreq(K, d=1.0 / K, device=DEV, dtype=F64) / L
        mz = torch.fft.rfftfreq(K, d=1.0 / K, device=DEV, dtype=F64) / L
        m2 = m[:, None, None] ** 2 + m[None, :, None] ** 2 + mz[None, None, :] ** 2
        m2[0, 0, 0] = 1.0
        g = COULOMB_F / (math.pi * L ** 3) * torch.exp(-math.pi ** 2 * m2 / _beta(1.0) ** 2) / m2
        g[0, 0, 0] = 0.0
        s["phi"] = (torch.fft.irfftn(torch.fft.rfftn(rho) * g, s=(K, K, K)) * K ** 3).float().contiguous()
    return s


def prepare(case, seed):
    kind = case["kind"]
    s = _inputs(case, seed)
    s["kind"] = kind
    n = s["n"]
    if kind in ("spread", "gather"):
        s["mesh"] = (case["K"],) * 3
        if kind == "spread":
            s["grid"] = torch.empty(s["mesh"], dtype=torch.float32, device=DEV)
        else:
            s["F"] = torch.empty((n, 3), dtype=torch.float32, device=DEV)
        return s
    s["rc"], s["beta"] = case["rc"], _beta(case["rc"])
    s["rlist"], s["r_inner"] = case.get("rlist"), case.get("r_inner")
    s["F"] = torch.empty((n, 3), dtype=torch.float32, device=DEV)
    s["E"] = None
    if kind == "batch":
        sizes = _sizes(case, seed)
        s["pl"] = nb.Pairlist.batch(np.concatenate([[0], 3 * np.cumsum(sizes)]), np.repeat(np.float32(s["edges"]), 3))
        s["E"] = torch.empty(2 * len(sizes), dtype=torch.float64, device=DEV)
        return s
    pl = s["pl"] = nb.Pairlist(n)
    if kind == "oneshot" or case.get("energy"):
        s["E"] = torch.empty(2, dtype=torch.float64, device=DEV)
    if kind == "halo":
        pl.set_home(s["n_home"])
    if kind == "forces" and case["coul"] != "ewald":
        pl.set_coulomb("rf" if case["coul"].startswith("rf") else "ewald", eps_rf=0.0, shift=case["coul"] == "ewald_shift",
                       excl_corr=case["coul"] == "rf_excl")
    if kind in ("forces", "adjoint", "halo"):
        pl.search(s["x"], s["box"], s["rlist"], s["eo"], s["ei"])
        pl.prune(s["x"], s["r_inner"])
    if kind == "adjoint":
        s["target"] = (100.0 * s["target_noise"]).float()
        s["g"] = torch.empty_like(s["target"])
    if kind == "cycle":
        s["Fs"] = [torch.empty((n, 3), dtype=torch.float32, device=DEV) for _ in s["frames"]]
    return s


def run(s):
    kind = s["kind"]
    if kind == "spread":
        nb.nb_pme_spread(s["x"], s["q"], s["box"], s["mesh"], s["grid"])
        return s["grid"]
    if kind == "gather":
        nb.nb_pme_gather(s["x"], s["q"], s["box"], s["mesh"], s["phi"], s["F"])
        return s["F"]
    pl, rc, beta, q, t, lj = s["pl"], s["rc"], s["beta"], s["q"], s["t"], s["lj"]
    if kind == "forces":
        pl.forces(s["frame"], q, t, lj, rc, beta, s["F"], s["E"], want_energy=False)
        return s["F"] if s["E"] is None else (s["F"], s["E"])
    if kind == "oneshot":
        pl.search(s["x"], s["box"], rc, s["eo"], s["ei"])
        pl.forces(s["x"], q, t, lj, rc, beta, s["F"], s["E"])
        return s["F"], s["E"]
    if kind == "cycle":
        frames = s["frames"]
        pl.search(frames[0], s["box"], s["rlist"], s["eo"], s["ei"])
        pl.prune(frames[0], s["r_inner"])
        for x, F in zip(frames, s["Fs"]):
            pl.forces(x, q, t, lj, rc, beta, F, want_energy=False)
        return s["Fs"]
    if kind == "adjoint":
        pl.forces(s["frame"], q, t, lj, rc, beta, s["F"], want_energy=False)
        torch.sub(s["F"], s["target"], out=s["g"])
        return (s["F"],) + pl.backward(s["frame"], q, t, lj, rc, beta, s["g"])
    if kind == "batch":
        pl.search(s["x"], None, s["rlist"], s["eo"], s["ei"])
        pl.prune(s["x"], rc)
        pl.forces(s["x"], q, t, lj, rc, beta, s["F"], s["E"])
        return s["F"], s["E"]
    pl.forces_part(nb.NB_PART_LOCAL, s["frame"], q, t, lj, rc, beta)
    pl.forces_part(nb.NB_PART_NONLOCAL, s["frame"], q, t, lj, rc, beta, s["F"])
    return s["F"]


# ---------------------------------------------------------------------------
# Necessary work
# ---------------------------------------------------------------------------

def work(case):
    """Bytes: each input read once and each output written once (per atom 12
    coordinates + 4 charge + 4 type + 12 force, exclusions where a search reads
    them, the mesh). Flops: 66 per pair within the cutoff (displacement, LJ,
    erfc, force), 42 for the reaction field, 136 more for the adjoint; the mesh
    steps 2 (spread) and 8 (gather) per mesh point of an atom's 64."""
    kind = case["kind"]
    n = 3 * sum(_sizes(case, 0))
    if kind in ("spread", "gather"):
        mesh = 4.0 * case["K"] ** 3
        return {"bytes": 16.0 * n + mesh + (12.0 * n if kind == "gather" else 0.0), "flops": 64.0 * n * (2 if kind == "spread" else 8)}
    pairs = n * 3 * DENSITY * (2.0 / 3.0) * math.pi * case["rc"] ** 3
    per_pair = 42.0 if case.get("coul", "").startswith("rf") else 66.0
    excl = 12.0 * n  # offsets and two partners per atom
    if kind == "cycle":
        return {"bytes": n * (8.0 + 24.0 * case["frames"]) + excl, "flops": per_pair * pairs * case["frames"]}
    if kind == "adjoint":
        return {"bytes": n * (20.0 + 12.0 + 12.0 + 16.0), "flops": (66.0 + 136.0) * pairs}
    return {"bytes": 32.0 * n + (excl if kind in ("oneshot", "batch") else 0.0), "flops": per_pair * pairs}


# ---------------------------------------------------------------------------
# The same in 64 bits
# ---------------------------------------------------------------------------

def _pair_blocks(x, L, rc):
    """The pairs i < j within rc of positions x [n, 3] in a cubic box of edge
    L, minimum image, in blocks (i, j, d = x_i - x_j)."""
    n = x.shape[0]
    m = int(L / rc)
    if m < 4 or n < 6000:
        rows = max(1, (1 << 25) // n)
        for a in range(0, n, rows):
            d = x[a:a + rows, None, :] - x[None, :, :]
            d -= L * torch.round(d / L)
            near = (d * d).sum(-1) < rc * rc
            near &= torch.arange(a, min(a + rows, n), device=DEV)[:, None] < torch.arange(n, device=DEV)[None, :]
            i, j = near.nonzero(as_tuple=True)
            yield i + a, j, d[i, j]
        return
    c = (x / L * m).long().clamp(0, m - 1)
    cid = (c[:, 0] * m + c[:, 1]) * m + c[:, 2]
    order = cid.argsort()
    count = torch.bincount(cid, minlength=m ** 3)
    first = count.cumsum(0) - count
    most = int(count.max())
    table = torch.full((m ** 3, most), -1, dtype=torch.int64, device=DEV)
    table[cid[order], torch.arange(n, device=DEV) - first[cid[order]]] = order
    cells = torch.arange(m ** 3, device=DEV)
    cx, cy, cz = cells // (m * m), (cells // m) % m, cells % m
    step = max(1, (1 << 25) // (most * most))
    for k in range(27):
        other = (((cx + k // 9 - 1) % m) * m + (cy + (k // 3) % 3 - 1) % m) * m + (cz + k % 3 - 1) % m
        for a in range(0, m ** 3, step):
            ti, tj = table[a:a + step], table[other[a:a + step]]
            d = x[ti.clamp(min=0)][:, :, None, :] - x[tj.clamp(min=0)][:, None, :, :]
            d -= L * torch.round(d / L)
            near = ((d * d).sum(-1) < rc * rc) & (ti[:, :, None] >= 0) & (ti[:, :, None] < tj[:, None, :])
            b, u, v = near.nonzero(as_tuple=True)
            yield ti[b, u], tj[b, v], d[b, u, v]


def _radial(r2, qq, c6, c12, rc, beta, coul, inside):
    """(energy LJ, energy Coulomb, -dE/dr / r) of pairs; ``inside``: the pair
    is of one molecule, which the list excludes."""
    ri2 = 1.0 / r2
    r = r2.sqrt()
    ri6 = ri2 ** 3
    out = ~inside
    e_lj = (c12 * ri6 * ri6 - c6 * ri6 - (c12 / rc ** 12 - c6 / rc ** 6)) * out
    s = (12 * c12 * ri6 * ri6 - 6 * c6 * ri6) * ri2 * out
    f = COULOMB_F * qq
    if coul.startswith("rf"):
        krf = 1.0 / (2 * rc ** 3)
        crf = 1.0 / rc + krf * rc * rc
        own = 1.0 if coul == "rf_excl" else 0.0
        w = out + own * inside
        e_c = f * ((krf * r2 - crf) * w + out / r)
        s = s + f * (out * ri2 / r - 2 * krf * w)
    else:
        a = torch.erfc(beta * r) / r
        e_c = f * (a - (math.erfc(beta * rc) / rc if coul == "ewald_shift" else 0.0)) * out
        s = s + f * (a + 2 * beta / math.sqrt(math.pi) * torch.exp(-(beta * r) ** 2)) * ri2 * out
    return e_lj, e_c, s


def _forces64(x, q, t, lj, L, rc, beta, coul="ewald"):
    x, q, lj, t = x.double(), q.double(), lj.double(), t.long()
    F = torch.zeros_like(x)
    E = torch.zeros(2, dtype=F64, device=DEV)
    for i, j, d in _pair_blocks(x, L, rc):
        c = lj[t[i], t[j]]
        e_lj, e_c, s = _radial((d * d).sum(-1), q[i] * q[j], c[:, 0], c[:, 1], rc, beta, coul, i // 3 == j // 3)
        E[0] += e_lj.sum()
        E[1] += e_c.sum()
        F.index_add_(0, i, s[:, None] * d)
        F.index_add_(0, j, -s[:, None] * d)
    return F, E


def _spline(x, K, L):
    """Mesh indices [n, 4] and weights M4, M4' [n, 4] along one axis."""
    u = x * (K / L)
    fl = torch.floor(u)
    w = (u - fl)[:, None] + torch.arange(4, device=DEV)  # argument of M4 at mesh points floor(u) - j
    k = (fl.long()[:, None] - torch.arange(4, device=DEV)) % K
    M = torch.where(w < 1, w ** 3 / 6, torch.where(w < 2, (-3 * (w - 1) ** 3 + 3 * (w - 1) ** 2 + 3 * (w - 1) + 1) / 6,
                    torch.where(w < 3, (3 * (w - 2) ** 3 - 6 * (w - 2) ** 2 + 4) / 6, (4 - w) ** 3 / 6)))
    D = torch.where(w < 1, w ** 2 / 2, torch.where(w < 2, (-3 * (w - 1) ** 2 + 2 * (w - 1) + 1) / 2,
                    torch.where(w < 3, (3 * (w - 2) ** 2 - 4 * (w - 2)) / 2, -(4 - w) ** 2 / 2)))
    return k, M, D


def exact(case, seed):
    kind = case["kind"]
    s = _inputs(case, seed)
    if kind in ("spread", "gather"):
        K, L = case["K"], float(np.float32(s["edges"][0]))
        x, q = s["x"].double(), s["q"].double()
        (kx, mx, dx), (ky, my, dy), (kz, mz, dz) = (_spline(x[:, a], K, L) for a in range(3))
        at = ((kx[:, :, None, None] * K + ky[:, None, :, None]) * K + kz[:, None, None, :]).reshape(-1, 64)
        outer = lambda a, b, c: (a[:, :, None, None] * b[:, None, :, None] * c[:, None, None, :]).reshape(-1, 64)  # noqa: E731
        if kind == "spread":
            grid = torch.zeros(K ** 3, dtype=F64, device=DEV)
            grid.index_add_(0, at.reshape(-1), (q[:, None] * outer(mx, my, mz)).reshape(-1))
            return grid.view(K, K, K)
        p = s["phi"].double().reshape(-1)[at]
        g = torch.stack([(outer(dx, my, mz) * p).sum(1), (outer(mx, dy, mz) * p).sum(1), (outer(mx, my, dz) * p).sum(1)], dim=1)
        return -q[:, None] * (K / L) * g
    rc, beta = float(np.float32(case["rc"])), float(np.float32(_beta(case["rc"])))
    if kind == "batch":
        sizes, F, E, a = _sizes(case, seed), [], [], 0
        for w, edge in zip(sizes, s["edges"]):
            b = a + 3 * w
            f, e = _forces64(s["x"][a:b], s["q"][a:b], s["t"][a:b], s["lj"], float(np.float32(edge)), rc, beta)
            F.append(f)
            E.append(e)
            a = b
        return torch.cat(F), torch.cat(E)
    L = s["box"][0]
    one = lambda x, coul="ewald": _forces64(x, s["q"], s["t"], s["lj"], L, rc, beta, coul)  # noqa: E731
    if kind == "cycle":
        return [one(x)[0] for x in s["frames"]]
    if kind == "oneshot":
        return one(s["x"])
    if kind == "halo":
        return one(s["frame"])[0]
    if kind == "forces":
        F, E = one(s["frame"], case["coul"])
        return (F, E) if case["energy"] else F
    # adjoint: the same forces with autograd, over all pairs at once
    x = s["frame"].double().requires_grad_(True)
    q = s["q"].double().requires_grad_(True)
    lj = s["lj"].double().requires_grad_(True)
    t = s["t"].long()
    blocks = [(i[k], j[k]) for i, j, _ in _pair_blocks(s["frame"].double(), L, rc) for k in [i // 3 != j // 3]]
    i, j = torch.cat([b[0] for b in blocks]), torch.cat([b[1] for b in blocks])
    d = x[i] - x[j]
    d = d - (L * torch.round(d / L)).detach()
    # the matrix is symmetric: each pair's derivative is shared by the entries (a, b) and (b, a)
    c = 0.5 * (lj[t[i], t[j]] + lj[t[j], t[i]])
    _, _, sc = _radial((d * d).sum(-1), q[i] * q[j], c[:, 0], c[:, 1], rc, beta, "ewald", torch.zeros_like(i, dtype=torch.bool))
    f = sc[:, None] * d
    F = torch.zeros_like(x).index_add(0, i, f).index_add(0, j, -f)
    target = (100.0 * s["target_noise"]).float().double()
    (0.5 * ((F - target) ** 2).sum()).backward()
    return F.detach(), x.grad, q.grad, lj.grad
