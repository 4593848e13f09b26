"""The calls that users of this library make, at the sizes they make them with.

Each case is one pass through the public Python entry points: molecular dynamics
(device and host arrays), single energy / force / virial evaluations, the
evaluation of a structure seen for the first time (list build included),
batched parameter fitting, and gradients of an energy-and-force loss. Inputs
are made on the GPU from a seed. ``exact`` restates Tersoff's definition in
plain torch, in 64 bits.
"""
import math

import numpy as np
import torch

import paper_1607_02904_gb300 as T

DEV = "cuda"
# Tersoff, Phys. Rev. B 39, 5566 (1989), Table I: A, B, lambda, mu, beta, n, c, d, h, R, S.
ELEM = {
    "Si": (1830.8, 471.18, 2.4799, 1.7322, 1.1e-6, 0.78734, 1.0039e5, 16.217, -0.59825, 2.7, 3.0),
    "C": (1393.6, 346.74, 3.4879, 2.2119, 1.5724e-7, 0.72751, 3.8049e4, 4.3484, -0.57058, 1.8, 2.1),
}
CHI_SIC = 0.9776
MASS = {"Si": 28.0855, "C": 12.011}  # amu
KB = 8.617333262e-5                  # eV / K
MVV2E = 1.0364269e-4                 # 1 amu A^2 / ps^2 in eV
AMU_G = 1.66053906660                # 1 amu / A^3 in g / cm^3
R_LIST = 4.0                         # the largest cutoff (3.0) and a skin of 1 A
DT = 0.001                           # ps
CELL_A = {"si": 5.432, "sic": 4.36}
SIGMA = {"si": 0.05, "sic": 0.08}    # Gaussian displacements, A
MIN_SEP, DENSITY = 1.8, 2.3          # random packings: A, g / cm^3


def listed():
    return [
        # A small cell run for long: every step is launch latency (thermo row at every step).
        dict(name="md_si216", kind="md", lattice="si", nx=3, ny=3, nz=3, fp64=False, steps=100, rebuild=-1, thermo=True),
        # The long accuracy run's cell: 32,000 atoms, energies at every step, rebuilds on half the skin.
        dict(name="md_si32k", kind="md", lattice="si", nx=20, ny=20, nz=10, fp64=False, steps=100, rebuild=-1, thermo=True),
        # The benchmark: 512,000 atoms at 1000 K, ten steps and a rebuild, mixed path.
        dict(name="md_si512k", kind="md", lattice="si", nx=40, ny=40, nz=40, fp64=False, steps=10, rebuild=10, thermo=False),
        # The same steps on the FP64 path.
        dict(name="md_si512k_fp64", kind="md", lattice="si", nx=40, ny=40, nz=40, fp64=True, steps=10, rebuild=10, thermo=False),
        # The same steps for a program that keeps its state in (pinned) host arrays.
        dict(name="md_host_si512k", kind="md_host", lattice="si", nx=40, ny=40, nz=40, fp64=False, steps=10, rebuild=10, thermo=False),
        # Production size: 16,384,000 atoms.
        dict(name="md_si16m", kind="md", lattice="si", nx=160, ny=160, nz=80, fp64=False, steps=20, rebuild=20, thermo=False),
        # One double-precision evaluation of a small cell (a reference value, a relaxation step).
        dict(name="eval_si4096_fp64", kind="eval", lattice="si", nx=8, ny=8, nz=8, fp64=True),
        # One evaluation of a large compound crystal.
        dict(name="eval_sic2m", kind="eval", lattice="sic", nx=64, ny=64, nz=64, fp64=False),
        # Screening: a structure's first evaluation, with its list build, at an odd size.
        dict(name="fresh_sic_odd", kind="fresh", lattice="sic", nx=23, ny=37, nz=29, fp64=False),
        # Fitting: energies, forces and the table gradient over 256 cells of uneven size.
        dict(name="fit_256", kind="fit", cells=256, nmin=64, nmax=4096, lam3=False, fp64=False),
        # A fitting iteration in double precision with the lambda3 term on: the table changes every time.
        dict(name="fit_step_fp64", kind="fit_step", cells=24, nmin=64, nmax=1024, lam3=True, fp64=True),
        # Gradients of an energy-and-force loss in the positions and the table, one crystal.
        dict(name="grad_si_odd", kind="grad", lattice="si", nx=31, ny=29, nz=37, fp64=False),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _crystal(rng, atoms_lo, atoms_hi, lattice):
    """Three edges in cubic cells (8 atoms each), unequal and odd as they fall; an edge is at least twice the list radius."""
    lo = 2 if lattice == "sic" else 3
    e = (_log_int(rng, atoms_lo, atoms_hi) / 8.0) ** (1.0 / 3.0)
    n = [max(lo, int(round(e * rng.uniform(0.75, 1.3)))) for _ in range(3)]
    return dict(lattice=lattice, nx=n[0], ny=n[1], nz=n[2])


def draw(rng):
    kind = rng.choice(["md", "md", "md", "md_host", "eval", "eval", "fresh", "fit", "fit_step", "grad"])
    fp64 = rng.random() < 0.4
    lattice = rng.choice(["si", "si", "sic"])
    if kind in ("md", "md_host"):
        c = _crystal(rng, 216, 400_000 if fp64 else 3_000_000, lattice)
        n = 8 * c["nx"] * c["ny"] * c["nz"]
        steps = max(5, min(100, _log_int(rng, 5, 100), (4_000_000 if fp64 else 40_000_000) // n))
        return dict(kind=kind, fp64=fp64, steps=steps, rebuild=rng.choice([-1, 10, 20]), thermo=rng.random() < 0.4, **c)
    if kind in ("eval", "fresh", "grad"):
        return dict(kind=kind, fp64=fp64, **_crystal(rng, 216, 400_000 if fp64 else 2_000_000, lattice))
    return dict(kind=kind, cells=_log_int(rng, 4, 48 if fp64 else 200), nmin=64, nmax=rng.choice([256, 1024, 3001]),
                lam3=rng.random() < 0.4, fp64=fp64)


# ---------------------------------------------------------------- inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(1607029040 + int(seed))


def _lattice(case, g):
    """Displaced diamond or zincblende crystal: x, types, box, species names."""
    a = CELL_A[case["lattice"]]
    fcc = torch.tensor([[0, 0, 0], [0, .5, .5], [.5, 0, .5], [.5, .5, 0]], dtype=torch.float64, device=DEV)
    basis = torch.cat([fcc, fcc + 0.25])
    r = [torch.arange(case[k], dtype=torch.float64, device=DEV) for k in ("nz", "ny", "nx")]
    z, y, x = torch.meshgrid(*r, indexing="ij")
    o = torch.stack([x.reshape(-1), y.reshape(-1), z.reshape(-1)], 1)
    pos = ((o[:, None, :] + basis) * a).reshape(-1, 3)
    pos += SIGMA[case["lattice"]] * torch.randn(pos.shape, dtype=torch.float64, device=DEV, generator=g)
    types = torch.zeros((o.shape[0], 8), dtype=torch.int32, device=DEV)
    names = ["Si"]
    if case["lattice"] == "sic":
        types[:, 4:] = 1
        names = ["Si", "C"]
    return pos.contiguous(), types.reshape(-1).contiguous(), np.array([case["nx"], case["ny"], case["nz"]]) * a, names


def _packings(case, g):
    """Random sequential insertion of Si/C atoms in periodic cubes, all cells at once: uneven counts, random C fraction up to 0.8.

    A voxel of edge at most MIN_SEP / sqrt(3) holds one atom at most, so the 125 voxels around a candidate hold
    every atom nearer than MIN_SEP. Of the candidates of one round the earlier one wins."""
    S = case["cells"]
    # the cells' sizes belong to the case, their contents to the seed
    sizes = np.random.default_rng([S, case["nmin"], case["nmax"]]).integers(case["nmin"], case["nmax"] + 1, S)
    n = torch.tensor(sizes, device=DEV)
    frac = 0.8 * torch.rand(S, device=DEV, generator=g, dtype=torch.float64)  # nearly pure C would be close to jamming
    sysid = torch.repeat_interleave(torch.arange(S, device=DEV), n)
    N = sysid.numel()
    types = (torch.rand(N, device=DEV, generator=g, dtype=torch.float64) < frac[sysid]).to(torch.int32)
    mass = torch.where(types == 1, MASS["C"], MASS["Si"]).double()
    L = (torch.zeros(S, dtype=torch.float64, device=DEV).index_add_(0, sysid, mass) * AMU_G / DENSITY).pow(1 / 3)
    L = L.clamp(min=2 * R_LIST + 1e-6)
    nv = torch.ceil(L * math.sqrt(3.0) / MIN_SEP).long()
    base = torch.cumsum(nv ** 3, 0) - nv ** 3
    total = int((nv ** 3).sum())
    k = torch.arange(-2, 3, device=DEV)
    off = torch.stack(torch.meshgrid(k, k, k, indexing="ij"), -1).reshape(-1, 3)
    pos = torch.zeros((N, 3), dtype=torch.float64, device=DEV)
    grid = torch.full((total,), -1, dtype=torch.long, device=DEV)
    pending = torch.arange(N, device=DEV)

    def near(at, vox, sys, table, places, mine=None):
        """Whether an entry of `table` (indices into places, -1 empty) is nearer than MIN_SEP (with mine: one of a lower index)."""
        hit = torch.zeros(at.shape[0], dtype=torch.bool, device=DEV)
        m, Ls = nv[sys][:, None], L[sys][:, None, None]
        for o in off.split(25):
            v = (vox[:, None, :] + o[None]) % m[:, :, None]
            q = table[base[sys][:, None] + (v[..., 2] * m + v[..., 1]) * m + v[..., 0]]
            d = places[q.clamp(min=0)] - at[:, None, :]
            d = d - Ls * torch.round(d / Ls)
            c = (q >= 0) & ((d * d).sum(-1) < MIN_SEP * MIN_SEP)
            if mine is not None:
                c &= q < mine[:, None]
            hit |= c.any(1)
        return hit

    for _ in range(1000):
        m = pending.numel()
        if not m:
            break
        atom = pending.repeat(max(1, 100_000 // m))  # many candidates an atom once few atoms are left
        sys = sysid[atom]
        at = torch.rand((atom.numel(), 3), dtype=torch.float64, device=DEV, generator=g) * L[sys][:, None]
        vox = torch.minimum((at / L[sys][:, None] * nv[sys][:, None]).long(), nv[sys][:, None] - 1)
        free = ~near(at, vox, sys, grid, pos)
        atom, at, vox, sys = atom[free], at[free], vox[free], sys[free]
        rank = torch.arange(atom.numel(), device=DEV)
        vid = base[sys] + (vox[:, 2] * nv[sys] + vox[:, 1]) * nv[sys] + vox[:, 0]
        first = torch.full((total,), atom.numel(), dtype=torch.long, device=DEV).scatter_reduce_(0, vid, rank, "amin")
        ok = first[vid] == rank
        first = torch.where(first == atom.numel(), -1, first)
        ok &= ~near(at, vox, sys, first, at, rank)
        best = torch.full((N,), atom.numel(), dtype=torch.long, device=DEV).scatter_reduce_(0, atom[ok], rank[ok], "amin")
        ok &= best[atom] == rank
        pos[atom[ok]] = at[ok]
        grid[vid[ok]] = atom[ok]
        pending = pending[best[pending] == atom.numel()]
    else:
        raise RuntimeError("a packing ran out of attempts")
    offsets = np.concatenate([[0], torch.cumsum(n, 0).cpu().numpy()]).astype(np.int32)
    return pos, types, offsets, np.repeat(L.cpu().numpy()[:, None], 3, 1)


def _velocities(types, names, g):
    """Maxwell velocities at 1000 K without net momentum, A / ps."""
    m = torch.tensor([MASS[s] for s in names], dtype=torch.float64, device=DEV)[types.long()][:, None]
    v = torch.randn((types.numel(), 3), dtype=torch.float64, device=DEV, generator=g) * torch.sqrt(KB * 1000.0 / (m * MVV2E))
    return v - (m * v).sum(0) / m.sum()


def _elements(names):
    chi = np.ones((len(names),) * 2)
    if len(names) == 2:
        chi[0, 1] = chi[1, 0] = CHI_SIC
    return np.array([ELEM[s] for s in names]), chi


def _loss_targets(n, sizes, g):
    """Reference energies and forces of a fit: cohesive energies about -4.3 eV an atom, forces of an eV / A."""
    e = -4.3 * sizes + 0.1 * sizes * torch.randn(sizes.shape, dtype=torch.float64, device=DEV, generator=g)
    return e, torch.randn((n, 3), dtype=torch.float64, device=DEV, generator=g)


def _inputs(case, seed):
    """The case's arrays, from the seed alone."""
    g = _gen(seed)
    if case["kind"] in ("fit", "fit_step"):
        x, types, offsets, boxes = _packings(case, g)
        names = ["Si", "C"]
        sizes = torch.tensor(np.diff(offsets), dtype=torch.float64, device=DEV)
        e_ref, f_ref = _loss_targets(x.shape[0], sizes, g)
        return dict(x=x, types=types, offsets=offsets, boxes=boxes, names=names, sizes=sizes, e_ref=e_ref, f_ref=f_ref)
    x, types, box, names = _lattice(case, g)
    d = dict(x=x, types=types, box=box, names=names)
    if case["kind"] in ("md", "md_host"):
        d["v"] = _velocities(types, names, g)
    if case["kind"] == "grad":
        d["sizes"] = torch.tensor(float(x.shape[0]), dtype=torch.float64, device=DEV)
        d["e_ref"], d["f_ref"] = _loss_targets(x.shape[0], d["sizes"], g)
    return d


def _library_table(names, lam3):
    t = T.mix_tersoff89(*_elements(names))
    if lam3:
        t = t.reshape(-1, T.NPARAM)
        t[:, T.FIELDS.index("lambda3")] = 1.7322
    return t.ravel()


def prepare(case, seed):
    s = dict(_inputs(case, seed), kind=case["kind"])
    prec = T.FP64 if case["fp64"] else T.MIXED
    table = _library_table(s["names"], case.get("lam3", False))
    n = s["x"].shape[0]
    if s["kind"] in ("fit", "fit_step", "grad"):
        s["table"] = torch.tensor(table, dtype=torch.float64, requires_grad=True)
        if s["kind"] == "grad":
            s["system"] = T.TersoffSystem(s["types"].cpu().numpy(), s["box"], R_LIST, prec)
            s["x"].requires_grad_(True)
        else:
            s["system"] = T.TersoffBatch(s["types"].cpu().numpy(), s["offsets"], s["boxes"], R_LIST, prec)
        with torch.no_grad():
            T.energy_forces(s["system"], s["x"], s["table"])  # uploads the table and builds the list
        return s
    ctx = s["ctx"] = T.Context(prec)
    ctx.params(table)
    s["e"] = torch.empty(1, dtype=torch.float64, device=DEV)
    s["f"] = torch.empty_like(s["x"])
    s["w"] = torch.empty(6, dtype=torch.float64, device=DEV)
    if s["kind"] == "fresh":
        return s
    ctx.neighbor_build(s["x"], s["types"], s["box"], R_LIST)
    if s["kind"] == "eval":
        return s
    ctx.compute(s["x"], None, s["f"])
    s["steps"], s["rebuild"] = case["steps"], case["rebuild"]
    s["mass"] = [MASS[q] for q in s["names"]]
    s["thermo"] = torch.empty((s["steps"], 3), dtype=torch.float64, device=DEV) if case["thermo"] else None
    if s["kind"] == "md_host":
        for k in ("x", "v", "f", "thermo"):
            if s[k] is not None:
                s[k] = s[k].cpu().pin_memory()
    return s


# ---------------------------------------------------------------- one pass
def _loss(s, e, f):
    return (((e - s["e_ref"]) / s["sizes"]) ** 2).mean() + ((f - s["f_ref"]) ** 2).mean()


def _relative_step(table, grad):
    """A fit's update: every entry moves by at most 1e-6 of itself, along the gradient."""
    rel = grad * table.detach()
    return table.detach() * (1.0 - 1e-6 * rel / rel.abs().max())


def run(s):
    k = s["kind"]
    if k in ("md", "md_host"):
        step = s["ctx"].md_step if k == "md" else s["ctx"].md_step_host
        step(s["x"], s["v"], s["f"], s["mass"], DT, s["steps"], s["rebuild"], s["thermo"])
        return {q: s[q] for q in ("x", "v", "f", "thermo") if s[q] is not None}
    if k in ("eval", "fresh"):
        if k == "fresh":
            s["ctx"].neighbor_build(s["x"], s["types"], s["box"], R_LIST)
        s["ctx"].compute(s["x"], s["e"], s["f"], s["w"])
        return {"energy": s["e"], "forces": s["f"], "virial": s["w"]}
    e, f = T.energy_forces(s["system"], s["x"], s["table"])
    loss = _loss(s, e, f)
    if k == "grad":
        gx, gt = torch.autograd.grad(loss, [s["x"], s["table"]])
        return {"loss": loss.detach(), "energy": e.detach(), "forces": f.detach(), "grad_x": gx, "grad_table": gt}
    (gt,) = torch.autograd.grad(loss, [s["table"]])
    out = {"loss": loss.detach(), "energies": e.detach(), "forces": f.detach(), "grad_table": gt}
    if k == "fit_step":
        with torch.no_grad():
            s["table"].copy_(_relative_step(s["table"], gt))
        out["table"] = s["table"].detach()
    return out


def _terms(case):
    """Atoms and bonds inside the cutoffs per atom (estimated for displaced compounds and packings)."""
    if "lattice" in case:
        return 8 * case["nx"] * case["ny"] * case["nz"], 4.0 if case["lattice"] == "si" else 5.4
    return case["cells"] * (case["nmin"] + case["nmax"]) / 2.0, 6.5


def work(case):
    n, z = _terms(case)
    # per bond its vector, length and share of the sums, per pair term and per three-body term (an FMA counts 2)
    flops = n * (36 * z + 63 * z + 61 * z * (z - 1))
    k = case["kind"]
    if k in ("md", "md_host"):
        return {"bytes": n * (2 * 72 + 4) + (24 * case["steps"] if case["thermo"] else 0), "flops": flops * case["steps"]}
    if k in ("eval", "fresh"):
        return {"bytes": n * (24 + 4 + 24), "flops": flops + (n * 30 * 15 if k == "fresh" else 0)}
    # x, species, targets read, forces written; the adjoint passes take about 2.5 (table) and 4 (positions) evaluations
    return {"bytes": n * (24 + 4 + 24 + 24 + (24 if k == "grad" else 0)), "flops": flops * (1 + 2.5 + (4 if k == "grad" else 0))}


# ---------------------------------------------------------------- the definition in 64 bits
def _exact_table(names, lam3):
    """(ns, ns, ns, 14) records m, gamma, lambda3, c, d, h, n, beta, lambda2, B, R, D, lambda1, A by Tersoff's mixing rules."""
    el, chi = _elements(names)
    A, B, lam, mu, be, n, c, d, h, Rin, Sout = el.T
    ns = len(names)
    t = np.zeros((ns, ns, ns, 14))
    for i in range(ns):
        for j in range(ns):
            for q in range(ns):
                R, S = math.sqrt(Rin[i] * Rin[q]), math.sqrt(Sout[i] * Sout[q])
                t[i, j, q] = (3, 1, 1.7322 if lam3 else 0, c[i], d[i], h[i], n[i], be[i], (mu[i] + mu[j]) / 2,
                              chi[i, j] * math.sqrt(B[i] * B[j]), (R + S) / 2, (S - R) / 2, (lam[i] + lam[j]) / 2,
                              math.sqrt(A[i] * A[j]))
    return torch.tensor(t, dtype=torch.float64, device=DEV)


def _near_pairs(x, box, rc):
    """Directed pairs (i, j) within rc (minimum image), sorted by i."""
    box = torch.as_tensor(box, dtype=torch.float64, device=DEV)
    n = x.shape[0]
    if n <= 4200:
        d = x[None, :, :] - x[:, None, :]
        d = d - box * torch.round(d / box)
        c = (d * d).sum(-1) <= rc * rc
        c.fill_diagonal_(False)
        return c.nonzero(as_tuple=True)
    nc = torch.floor(box / rc).long()
    w = x - box * torch.floor(x / box)
    c3 = torch.minimum((w / box * nc).long(), nc - 1)
    cid = (c3[:, 2] * nc[1] + c3[:, 1]) * nc[0] + c3[:, 0]
    count = torch.bincount(cid, minlength=int(nc.prod()))
    order = torch.argsort(cid, stable=True)
    rank = torch.arange(n, device=DEV) - (torch.cumsum(count, 0) - count)[cid[order]]
    members = torch.full((count.numel(), int(count.max())), -1, dtype=torch.long, device=DEV)
    members[cid[order], rank] = order
    ii, jj = [], []
    me = torch.arange(n, device=DEV)[:, None]
    for a in (-1, 0, 1):
        for b in (-1, 0, 1):
            for e in (-1, 0, 1):
                o = (c3 + torch.tensor([a, b, e], device=DEV)) % nc
                q = members[(o[:, 2] * nc[1] + o[:, 1]) * nc[0] + o[:, 0]]
                d = x[q.clamp(min=0)] - x[:, None, :]
                d = d - box * torch.round(d / box)
                keep = (q >= 0) & (q != me) & ((d * d).sum(-1) <= rc * rc)
                i, s = keep.nonzero(as_tuple=True)
                ii.append(i)
                jj.append(q[i, s])
    i, j = torch.cat(ii), torch.cat(jj)
    o = torch.argsort(i, stable=True)
    return i[o], j[o]


def _taper(r, R, D):
    inner, outer = r <= R - D, r >= R + D
    s = torch.sin((math.pi / 4) * (R + D - r) / D) ** 2
    return torch.where(inner, torch.ones_like(r), torch.where(outer, torch.zeros_like(r), s))


def _pair_energies(d, i, j, types, tab, n):
    """V of every directed pair with bond vector d (i ascending): 1/2 f_C (f_R + b f_A)."""
    r = torch.linalg.norm(d, dim=1)
    u = d / r[:, None]
    z = torch.bincount(i, minlength=n)
    start = torch.cumsum(z, 0) - z
    Z = max(1, int(z.max()))
    at = torch.arange(Z, device=DEV)
    K = start[i][:, None] + at  # the pairs of the same centre
    me = torch.arange(i.numel(), device=DEV)[:, None]
    valid = (at < z[i][:, None]) & (K != me)
    K = torch.where(valid, K, me)
    ti, tj = types[i], types[j]
    p3 = lambda q: tab[ti[:, None], tj[:, None], types[j[K]], q]  # noqa: E731
    p2 = lambda q: tab[ti, tj, tj, q]  # noqa: E731
    rk = r[K]
    t = p3(5) - (u[:, None, :] * u[K]).sum(-1)
    c2, d2 = p3(3) ** 2, p3(4) ** 2
    term = _taper(rk, p3(10), p3(11)) * p3(1) * (1 + c2 * t * t / (d2 * (d2 + t * t)))
    if bool((tab[..., 2] != 0).any()):
        term = term * torch.exp((p3(2) * (r[:, None] - rk)) ** 3)  # m = 3 throughout
    zeta = torch.where(valid, term, torch.zeros_like(term)).sum(1)
    some = zeta > 0
    u_ = (p2(7) * torch.where(some, zeta, torch.ones_like(zeta))) ** p2(6)
    b = torch.where(some, (1 + u_) ** (-1 / (2 * p2(6))), torch.ones_like(zeta))
    return 0.5 * _taper(r, p2(10), p2(11)) * (p2(13) * torch.exp(-p2(12) * r) - b * p2(9) * torch.exp(-p2(8) * r))


def _evaluate(x, types, box, tab, pairs, chunk=1 << 18):
    """Energy, forces and virial over the given pairs, centre atoms taken `chunk` at a time."""
    box = torch.as_tensor(box, dtype=torch.float64, device=DEV)
    i, j = pairs
    n, E = x.shape[0], 0.0
    d = x[j] - x[i]
    d = d - box * torch.round(d / box)
    keep = (d * d).sum(1) < 3.0 ** 2
    i, j, d = i[keep], j[keep], d[keep]
    F, W = torch.zeros_like(x), torch.zeros(3, 3, dtype=torch.float64, device=DEV)
    for a in range(0, n, chunk):
        lo, hi = (int(torch.searchsorted(i, torch.tensor(q, device=DEV))) for q in (a, min(n, a + chunk)))
        if lo == hi:
            continue
        dl = d[lo:hi].detach().requires_grad_(True)
        V = _pair_energies_of(dl, i[lo:hi], j[lo:hi], types, tab, a, min(n, a + chunk))
        (gd,) = torch.autograd.grad(V, dl)
        F.index_add_(0, i[lo:hi], gd)
        F.index_add_(0, j[lo:hi], -gd)
        W -= dl.detach().T @ gd
        E += float(V.detach())
    return E, F, torch.stack([W[0, 0], W[1, 1], W[2, 2], W[0, 1], W[0, 2], W[1, 2]])


def _pair_energies_of(d, i, j, types, tab, a, b):
    """The summed energy of the centres a .. b - 1."""
    r = torch.cat([types[a:b], types[j]])  # local numbering: the centres, then every pair's neighbour
    m = b - a
    return _pair_energies(d, i - a, m + torch.arange(j.numel(), device=DEV), r, tab, m).sum()


def _exact_md(case, s, tab):
    types, box = s["types"].long(), torch.as_tensor(s["box"], dtype=torch.float64, device=DEV)
    m = torch.tensor([MASS[q] for q in s["names"]], dtype=torch.float64, device=DEV)[types][:, None]
    x, v = s["x"].clone(), s["v"].clone()
    pairs = _near_pairs(x, s["box"], R_LIST)
    _, f, _ = _evaluate(x, types, box, tab, pairs)
    rows = []
    for step in range(case["steps"]):
        v = v + 0.5 * DT / MVV2E * f / m
        x = x + DT * v
        if step % 10 == 9:
            pairs = _near_pairs(x, s["box"], R_LIST)
        e, f, _ = _evaluate(x, types, box, tab, pairs)
        v = v + 0.5 * DT / MVV2E * f / m
        if case["thermo"]:
            ke = float(0.5 * MVV2E * (m * v * v).sum())
            rows.append((e, ke, e + ke))
    out = {"x": x, "v": v, "f": f}
    if case["thermo"]:
        out["thermo"] = torch.tensor(rows, dtype=torch.float64)
    return out


def exact(case, seed):
    n, _ = _terms(case)
    if case["kind"] in ("md", "md_host") and n * case["steps"] > 3e7:
        return None
    s = _inputs(case, seed)
    types = s["types"].long()
    tab = _exact_table(s["names"], case.get("lam3", False))
    if case["kind"] in ("md", "md_host"):
        return _exact_md(case, s, tab)
    if case["kind"] in ("eval", "fresh"):
        e, f, w = _evaluate(s["x"], types, s["box"], tab, _near_pairs(s["x"], s["box"], 3.0))
        return {"energy": torch.tensor([e], dtype=torch.float64), "forces": f, "virial": w}
    if case["kind"] == "grad":
        if n > 400_000:
            return None
        off, boxes = [0, s["x"].shape[0]], [s["box"]]
    else:
        off, boxes = s["offsets"].tolist(), s["boxes"]
    i, j, sh = [], [], []
    for q, box in enumerate(boxes):
        a, b = _near_pairs(s["x"][off[q]:off[q + 1]], box, 3.0)
        i.append(a + off[q])
        j.append(b + off[q])
        L = torch.as_tensor(box, dtype=torch.float64, device=DEV)
        sh.append(L * torch.round((s["x"][j[-1]] - s["x"][i[-1]]) / L))
    i, j, sh = torch.cat(i), torch.cat(j), torch.cat(sh)
    x, tab = s["x"].requires_grad_(True), tab.requires_grad_(True)
    V = _pair_energies(x[j] - x[i] - sh, i, j, types, tab, x.shape[0])
    sysid = torch.repeat_interleave(torch.arange(len(boxes), device=DEV), torch.tensor(np.diff(off), device=DEV))
    e = torch.zeros(len(boxes), dtype=torch.float64, device=DEV).index_add(0, sysid[i], V)
    if case["kind"] == "grad":
        e = e.reshape(())
    f = -torch.autograd.grad(e.sum(), x, create_graph=True)[0]
    loss = _loss(s, e, f)
    if case["kind"] == "grad":
        gx, gt = torch.autograd.grad(loss, [x, tab])
        return {"loss": loss.detach(), "energy": e.detach(), "forces": f.detach(), "grad_x": gx, "grad_table": gt.reshape(-1).cpu()}
    (gt,) = torch.autograd.grad(loss, [tab])
    gt = gt.reshape(-1).cpu()
    out = {"loss": loss.detach(), "energies": e.detach(), "forces": f.detach(), "grad_table": gt}
    if case["kind"] == "fit_step":
        out["table"] = _relative_step(tab.detach().reshape(-1).cpu(), gt)
    return out
