"""Performance cases: what a user of this library has it do.

Every case is one call (or one relaxation) through the public Python binding
of the C ABI.  Systems are seeded synthetic ones of the shapes this
repository's benchmark and tests use: Cu (second-moment EAM) boxes, slabs and
batches, the Lennard-Jones vacancy box, diamond Si (Stillinger-Weber), the Cu
vacancy hop as a nudged elastic band.  Units: eV, Angstrom, ps (LJ: reduced).

``exact`` restates the same mathematics (energies by formula, forces and
Hessian products by torch.autograd, FIRE 2.0 step by step, the conjugate
gradient solve) in plain 64-bit torch.
"""
from __future__ import annotations

import itertools
import math

import torch

import paper_1908_02038_gb300 as fg

F64 = torch.float64

# potentials and integration settings of the benchmark's workloads
CU = dict(A=0.0855, xi=1.224, p=10.96, q=2.278, r0=2.556, rs=4.5, rc=5.0)
CU_A, CU_MASS, CU_DT = 3.615, 63.546 / 9648.533212331001, 0.001
LJ = dict(eps=1.0, sigma=1.0, rc_lj=2.5)
LJ_A, LJ_MASS, LJ_DT = 1.5874, 1.0, 0.005
SI = dict(eps=2.1683, sigma=2.0951, sw_A=7.049556277, sw_B=0.6022245584, sw_p=4.0, sw_q=0.0,
          sw_a=1.80, sw_lambda=21.0, sw_gamma=1.20)
SI_A = 4.0 * 2.0 ** (1.0 / 6.0) * SI["sigma"] / math.sqrt(3.0)
SI_MASS, SI_DT = 28.0855 / 9648.533212331001, 0.001
THETA = [CU["A"], CU["xi"], CU["p"], CU["q"]]
SKIN = 0.3

FCC = [[0, 0, 0], [.5, .5, 0], [.5, 0, .5], [0, .5, .5]]
DIAMOND = FCC + [[.25, .25, .25], [.75, .75, .25], [.75, .25, .75], [.25, .75, .75]]


# ---------------------------------------------------------------------------
# the cases

def listed():
    return [
        # one force evaluation of a small periodic cell, as a caller's own
        # integrator or line search asks for it: latency
        dict(name="cu497_eval", do="eval", pot="cu", form="fp64", nx=5, ny=5, nz=5, vac=3,
             noise=0.05, slab=False),
        # the same for a plug-in that may not allocate (all pairs, static scratch)
        dict(name="cu4k_noalloc", do="noalloc", pot="cu", nx=10, ny=10, nz=10, vac=40, noise=0.05),
        # one evaluation of a mid-size free-standing film with an odd number of
        # layers (open axis, uneven cells)
        dict(name="cu120k_slab_eval", do="eval", pot="cu", form="fp64", nx=32, ny=31, nz=30,
             vac=17, noise=0.05, slab=True),
        # the smallest relaxation: the LJ vacancy box to a tight force
        dict(name="lj255_relax", do="relax", pot="lj", form="fp64", nx=4, ny=4, nz=4, vac=1,
             noise=0.1, ftol=1e-6, maxiter=400, steps=171),
        # small and ordinary Cu vacancy boxes (1 % vacancies)
        dict(name="cu4k_relax", do="relax", pot="cu", form="fp64", nx=10, ny=10, nz=10, vac=40,
             noise=0.05, ftol=1e-4, maxiter=400, steps=133),
        dict(name="cu32k_relax", do="relax", pot="cu", form="fp64", nx=20, ny=20, nz=20, vac=320,
             noise=0.05, ftol=1e-4, maxiter=400, steps=143),
        # the headline box: 63^3 cells, 2 % strain, a 20 A void, in the default
        # form and in the FP32-pair form (which finishes in FP64)
        dict(name="cu1m_relax", do="relax", pot="cu", form="fp64", nx=63, ny=63, nz=63, vac=0,
             void=20.0, strain=0.02, noise=0.02, ftol=1e-2, maxiter=400, steps=73),
        dict(name="cu1m_relax_fp32pair", do="relax", pot="cu", form="fp32", nx=63, ny=63, nz=63,
             vac=0, void=20.0, strain=0.02, noise=0.02, ftol=1e-2, maxiter=400, steps=73),
        # the three-body potential: five vacancies in a Si slab
        dict(name="si33k_slab_relax", do="relax", pot="si", form="fp64", nx=16, ny=16, nz=16,
             vac=5, noise=0.05, slab=True, ftol=1e-2, maxiter=400, steps=66),
        # an ensemble of defect boxes of uneven size in one launch
        dict(name="batch512_fp32pair", do="batch", form="fp32", n_sys=512, nmin=3, nmax=12,
             noise=0.05, ftol=1e-3, maxiter=400, steps=97),
        # a transition path: 6 movable images of the vacancy hop, climbing
        dict(name="neb6x6911_relax", do="neb", nx=12, n_img=6, noise=0.01, ftol=1e-6, maxiter=60,
             steps=60),
        # backward of a relaxation in the potential's parameters
        dict(name="cu32k_implicit_grad", do="implicit", nx=20, ny=20, nz=20, vac=1, noise=0.002,
             steps=199),
    ]


def draw(rng):
    """One more case of the same ranges: a kind, an option, and sizes spread
    over the logarithm of the atom count."""
    def cells(lo, hi, per_cell=4):
        # a box of about exp(U) atoms, with unequal edges
        n = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        e = (n / per_cell) ** (1.0 / 3.0)
        return [max(3, min(63, int(round(e * rng.uniform(0.85, 1.15))))) for _ in range(3)]

    kind = rng.choice(["relax", "relax", "relax", "relax32", "lj", "si", "eval", "eval", "noalloc",
                       "batch", "neb", "energy_grad", "hvp", "implicit"])
    if kind in ("relax", "relax32"):
        nx, ny, nz = cells(300, 700_000)
        it = rng.randint(20, 60)
        return dict(do="relax", pot="cu", form="fp64" if kind == "relax" else "fp32", nx=nx, ny=ny,
                    nz=nz, vac=max(1, int(0.01 * 4 * nx * ny * nz * rng.random())),
                    noise=round(rng.uniform(0.02, 0.06), 3), slab=rng.random() < 0.3, ftol=1e-6,
                    maxiter=it, steps=it)
    if kind == "lj":
        it = rng.randint(40, 200)
        return dict(do="relax", pot="lj", form="fp64", nx=rng.randint(4, 9), ny=rng.randint(4, 9),
                    nz=rng.randint(4, 16), vac=rng.randint(1, 5), noise=round(rng.uniform(0.05, 0.1), 3),
                    ftol=1e-7, maxiter=it, steps=it)
    if kind == "si":
        nx, ny, nz = cells(500, 60_000, 8)
        it = rng.randint(20, 60)
        return dict(do="relax", pot="si", form="fp64", nx=nx, ny=ny, nz=nz, vac=rng.randint(1, 9),
                    noise=round(rng.uniform(0.02, 0.06), 3), slab=rng.random() < 0.5, ftol=1e-6,
                    maxiter=it, steps=it)
    if kind == "eval":
        nx, ny, nz = cells(200, 700_000)
        return dict(do="eval", pot="cu", form=rng.choice(["fp64", "fp64", "fp64_full", "analytic", "fp32"]),
                    nx=nx, ny=ny, nz=nz, vac=rng.randint(1, 3 + nx * ny * nz // 50),
                    noise=round(rng.uniform(0.02, 0.06), 3), slab=rng.random() < 0.4)
    if kind == "noalloc":
        if rng.random() < 0.3:
            return dict(do="noalloc", pot="lj", nx=rng.randint(4, 10), ny=rng.randint(4, 10),
                        nz=rng.randint(4, 10), vac=rng.randint(1, 5), noise=0.1)
        nx, ny, nz = cells(200, 24_000)
        return dict(do="noalloc", pot="cu", nx=nx, ny=ny, nz=nz, vac=rng.randint(1, 9), noise=0.05)
    if kind == "batch":
        lo = rng.randint(3, 7)
        it = rng.randint(20, 60)
        return dict(do="batch", form=rng.choice(["fp32", "fp64"]), n_sys=int(math.exp(rng.uniform(2.5, 6.0))),
                    nmin=lo, nmax=rng.randint(lo + 1, 12), noise=0.05, ftol=1e-6, maxiter=it, steps=it)
    if kind == "neb":
        it = rng.randint(15, 50)
        return dict(do="neb", nx=rng.randint(4, 12), n_img=rng.randint(3, 8), noise=0.01, ftol=1e-6,
                    maxiter=it, steps=it)
    nx, ny, nz = cells(300, 40_000 if kind == "implicit" else 200_000)
    return dict(do=kind, nx=nx, ny=ny, nz=nz, vac=rng.randint(1, 3),
                noise=0.002 if kind == "implicit" else 0.03, steps=150)


def work(case):
    """Bytes: positions read and results written once.  Operations: the
    method's floating-point work per pair inside the cut-off and evaluation
    (the density and force passes of the Cu potential 95 per pair, LJ 31, the
    Si pair and triplet terms 480 per atom, a Hessian product 60 per pair)."""
    if case["do"] == "batch":
        cells = [n ** 3 for n in range(case["nmin"], case["nmax"] + 1)]
        n = 4 * case["n_sys"] * sum(cells) / len(cells)
    elif case["do"] == "neb":
        n = (4 * case["nx"] ** 3 - 1) * case["n_img"]
    else:
        n = (8 if case.get("pot") == "si" else 4) * case["nx"] * case["ny"] * case["nz"] - case["vac"]
    per_atom = {"si": 480.0, "lj": 23 * 31.0}.get(case.get("pot"), 21 * 95.0)
    if case["do"] in ("hvp", "implicit"):
        per_atom = 21 * 60.0
    once = case["do"] in ("eval", "noalloc", "energy_grad", "hvp")
    evals = 1 if once else case["steps"] + 1
    vectors = {"hvp": 3, "implicit": 3}.get(case["do"], 2)
    return {"bytes": 24.0 * vectors * n, "flops": per_atom * n * evals}


# ---------------------------------------------------------------------------
# inputs

def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _sites(nx, ny, nz, a, basis):
    g = torch.stack(torch.meshgrid(*(torch.arange(n, device="cuda", dtype=F64) for n in (nx, ny, nz)),
                                   indexing="ij"), -1).reshape(-1, 1, 3)
    return ((g + torch.tensor(basis, device="cuda", dtype=F64)) * a).reshape(-1, 3)


def _system(case, seed):
    """Lattice with vacancies (and strain, a void, vacuum above a slab) and
    displacement noise: positions, box, periodic flags, lattice sites, first
    vacant site."""
    pot = case.get("pot", "cu")
    a = {"cu": CU_A, "lj": LJ_A, "si": SI_A}[pot]
    nc = [case["nx"], case["ny"], case["nz"]]
    gen = _gen(seed)
    x = _sites(*nc, a, DIAMOND if pot == "si" else FCC)
    box = [n * a for n in nc]
    if case.get("strain"):
        x[:, 0] *= 1.0 + case["strain"]
        box[0] *= 1.0 + case["strain"]
    keep = torch.ones(len(x), dtype=torch.bool, device="cuda")
    vacant = None
    if case.get("void"):
        keep &= ((x - torch.tensor(box, device="cuda", dtype=F64) / 2) ** 2).sum(1) >= case["void"] ** 2
    if case["vac"]:
        out = torch.randperm(len(x), generator=gen, device="cuda")[:case["vac"]]
        keep[out] = False
        vacant = x[out[0]].clone()
    x = x[keep].contiguous()
    if pot == "lj":   # uniform, as the LJ workload's recipe
        noise = (2.0 * torch.rand(x.shape, generator=gen, device="cuda", dtype=F64) - 1.0) * case["noise"]
    else:
        noise = torch.randn(x.shape, generator=gen, device="cuda", dtype=F64) * case["noise"]
    periodic = (1, 1, 1)
    if case.get("slab"):
        box[2] += 10.0
        periodic = (1, 1, 0)
    return x + noise, box, periodic, x, vacant


def _batch(case, seed):
    """Uneven Cu boxes with 1 to 3 vacancies each: packed positions, boxes,
    counts.  The sizes belong to the case, the vacancies and the noise to the seed."""
    gen = _gen(seed)
    host = torch.Generator().manual_seed(int(seed))
    size = torch.Generator().manual_seed(case["n_sys"])
    xs, boxes = [], []
    lattice = {}
    for _ in range(case["n_sys"]):
        n = int(torch.randint(case["nmin"], case["nmax"] + 1, (1,), generator=size))
        k = int(torch.randint(1, 4, (1,), generator=size))
        if n not in lattice:
            lattice[n] = _sites(n, n, n, CU_A, FCC)
        keep = torch.randperm(4 * n ** 3, generator=host)[k:].sort().values
        xs.append(lattice[n][keep.cuda()])
        boxes.append([n * CU_A] * 3)
    x = torch.cat(xs)
    x = x + torch.randn(x.shape, generator=gen, device="cuda", dtype=F64) * case["noise"]
    return x, boxes, [len(v) for v in xs]


def _path(case, seed):
    """Straight-line path of a nearest-neighbour vacancy hop in a Cu box."""
    gen = _gen(seed)
    n = case["nx"]
    x = _sites(n, n, n, CU_A, FCC)
    L = n * CU_A
    v = int(torch.randint(len(x), (1,), generator=gen, device="cuda"))
    d = x - x[v]
    d = d - L * torch.round(d / L)
    near = torch.nonzero((d.norm(dim=1) - CU_A / math.sqrt(2)).abs() < 1e-6).reshape(-1)
    w = int(near[torch.randint(len(near), (1,), generator=gen, device="cuda")])
    keep = torch.arange(len(x), device="cuda") != v
    t = torch.linspace(0, 1, case["n_img"] + 2, device="cuda", dtype=F64)[:, None, None]
    move = torch.zeros_like(x)
    move[w] = -d[w]
    noise = torch.randn(x.shape, generator=gen, device="cuda", dtype=F64) * case["noise"]
    return (x + noise + t * move)[:, keep].contiguous(), [L] * 3


def _potential(pot, form="fp64"):
    if pot == "lj":
        return fg.Potential(fg.FIRE_POT_LJ, skin=SKIN, **LJ)
    if pot == "si":
        return fg.Potential(fg.FIRE_POT_SW, skin=SKIN, **SI)
    return fg.Potential(fg.FIRE_POT_RGL, skin=SKIN, **CU,
                        precision=fg.FIRE_PREC_FP32_PAIR if form == "fp32" else fg.FIRE_PREC_FP64,
                        pair_eval=fg.FIRE_PAIR_ANALYTIC if form in ("analytic", "fp32") else fg.FIRE_PAIR_TABLE,
                        newton=fg.FIRE_NEWTON_OFF if form == "fp64_full" else fg.FIRE_NEWTON_AUTO)


def _mass_dt(pot):
    return {"cu": (CU_MASS, CU_DT), "lj": (LJ_MASS, LJ_DT), "si": (SI_MASS, SI_DT)}[pot]


def _loss_gradient(x, sites, vacant, box):
    """dL/dx of L = sum |x_i - site_i|^2 over the atoms within 6 A of the vacancy."""
    L = torch.tensor(box, device="cuda", dtype=F64)
    d = sites - vacant
    d = d - L * torch.round(d / L)
    return 2.0 * (x - sites) * (d.norm(dim=1, keepdim=True) < 6.0)


def prepare(case, seed):
    do, pot = case["do"], case.get("pot", "cu")
    mass, dt = _mass_dt(pot)
    if do == "batch":
        x, boxes, counts = _batch(case, seed)
        h = fg.FireBatch(counts, mass, _potential("cu", case["form"]), dt_start=dt)
        h.set_tuning(1024, 1)   # the launch shape the autotuner settles on for such batches
        return dict(case=case, x=x, box=boxes, h=h)
    if do == "neb":
        x, box = _path(case, seed)
        h = fg.FireNEB(case["n_img"], x.shape[1], mass, _potential("cu"), 1.0, True, dt_start=dt)
        return dict(case=case, x=x, box=box, h=h)
    x, box, periodic, sites, vacant = _system(case, seed)
    s = dict(case=case, x=x, box=box, periodic=periodic)
    if do == "noalloc":
        s["pot"] = _potential(pot).c()
        return s
    s["h"] = fg.FireHandle(len(x), mass, _potential(pot, case.get("form", "fp64")), periodic=periodic,
                           dt_start=dt)
    if do == "hvp":
        s["u"] = torch.randn(x.shape, generator=_gen(seed + 1), device="cuda", dtype=F64)
    if do == "implicit":
        s["u"] = _loss_gradient(x, sites, vacant, box)
    return s


def run(state):
    case, x, box = state["case"], state["x"], state["box"]
    do = case["do"]
    if do == "relax":
        x = x.clone()
        r = state["h"].minimize_dev(x, box, case["ftol"], case["maxiter"])
        return {"x": x, "energy": r.energy}
    if do == "batch":
        x = x.clone()
        r = state["h"].minimize_dev(x, box, case["ftol"], case["maxiter"])
        return {"x": x, "energy": torch.tensor([v.energy for v in r], dtype=F64)}
    if do == "neb":
        x = x.clone()
        _, energies, _ = state["h"].minimize_dev(x, box, case["ftol"], case["maxiter"])
        return {"x": x, "energy": energies}
    out = torch.empty_like(x)
    if do in ("eval", "noalloc"):
        energy = torch.empty(1, device="cuda", dtype=F64)
        if do == "eval":
            fg.fire_energy_forces_dev(state["h"].h, x, box, out, energy)
        else:
            fg.fire_energy_forces_noalloc(state["pot"], x, box, state["periodic"], out, energy)
        return {"forces": out, "energy": energy}
    if do == "energy_grad":
        energy, theta = fg.fire_rgl_energy_grad_dev(state["h"].h, x, box, THETA, out)
        return {"forces": out, "energy": energy, "theta": theta}
    if do == "hvp":
        fg.fire_rgl_hvp_dev(state["h"].h, x, box, THETA, state["u"], out)
        return {"hu": out}
    theta, _ = fg.fire_rgl_implicit_grad_dev(state["h"].h, x, box, THETA, state["u"], d_lambda=out)
    return {"theta": theta, "lambda": out}


# ---------------------------------------------------------------------------
# the same results in plain 64-bit torch

def _all_pairs(x, L, per, rl):
    """Index pairs i < j closer than rl (minimum image), row block by row block."""
    n, got = len(x), []
    step = max(1, 20_000_000 // n)
    for lo in range(0, n, step):
        d = x[None, :, :] - x[lo:lo + step, None, :]
        d = d - L * torch.round(d / L) * per
        m = (d * d).sum(-1) < rl * rl
        m &= torch.arange(n, device="cuda") > torch.arange(lo, min(n, lo + step), device="cuda")[:, None]
        i, j = torch.nonzero(m, as_tuple=True)
        got.append(torch.stack([i + lo, j]))
    return torch.cat(got, 1)


def _cell_pairs(x, L, per, rl):
    """The same through cells at least rl wide (three or more on a periodic axis)."""
    nc = torch.floor(L / rl).long().clamp(min=1)
    c = torch.floor(torch.where(per > 0, x - L * torch.floor(x / L), x) / L * nc).long()
    c = torch.minimum(c.clamp(min=0), nc - 1)
    dims = nc.tolist()
    ncell = dims[0] * dims[1] * dims[2]
    cid = (c[:, 0] * dims[1] + c[:, 1]) * dims[2] + c[:, 2]
    order = torch.argsort(cid, stable=True)
    count = torch.bincount(cid, minlength=ncell)
    start = torch.cumsum(count, 0) - count
    m = int(count.max())
    table = torch.full((ncell + 1, m), -1, dtype=torch.long, device="cuda")
    table[cid[order], torch.arange(len(x), device="cuda") - start[cid[order]]] = order
    grid = torch.stack(torch.meshgrid(*(torch.arange(k, device="cuda") for k in dims), indexing="ij"),
                       -1).reshape(-1, 3)
    got = []
    for o in itertools.product((-1, 0, 1), repeat=3):
        if o < (0, 0, 0):
            continue   # each pair of cells once
        nb = grid + torch.tensor(o, device="cuda")
        inside = ((nb >= 0) & (nb < nc) | (per > 0)).all(1)
        nb = nb % nc
        nid = torch.where(inside, (nb[:, 0] * dims[1] + nb[:, 1]) * dims[2] + nb[:, 2], ncell)
        step = max(1, 20_000_000 // (m * m))
        for lo in range(0, ncell, step):
            a, b = table[lo:min(ncell, lo + step), :, None], table[nid[lo:lo + step]][:, None, :]
            ok = (a >= 0) & (b >= 0)
            if o == (0, 0, 0):
                ok &= a < b
            k = torch.nonzero(ok.reshape(-1)).reshape(-1)
            i, j = a.expand(ok.shape).reshape(-1)[k], b.expand(ok.shape).reshape(-1)[k]
            d = x[j] - x[i]
            d = d - L * torch.round(d / L) * per
            near = (d * d).sum(1) < rl * rl
            got.append(torch.stack([i[near], j[near]]))
    return torch.cat(got, 1)


class _Model:
    """Energies of packed systems from a pair list with a wide skin."""

    def __init__(self, pot, x, boxes, counts, periodic, skin=0.9):
        self.pot, self.counts = pot, counts
        self.per = torch.tensor(periodic, device="cuda", dtype=F64)
        self.boxes = torch.tensor(boxes, device="cuda", dtype=F64).reshape(-1, 3)
        self.S = len(counts)
        self.sys = torch.repeat_interleave(torch.arange(self.S, device="cuda"),
                                           torch.tensor(counts, device="cuda"))
        self.rc = {"cu": CU["rc"], "lj": LJ["rc_lj"], "si": SI["sw_a"] * SI["sigma"]}[pot]
        self.skin = skin if pot != "lj" else 0.5
        self.theta = torch.tensor(THETA, device="cuda", dtype=F64)
        self.ref = None
        self.relist(x)

    def relist(self, x):
        if self.ref is not None and float((x - self.ref).norm(dim=1).max()) < 0.5 * self.skin:
            return
        self.ref, lists, off = x.clone(), [], 0
        for s, n in enumerate(self.counts):
            L, rl, y = self.boxes[s], self.rc + self.skin, x[off:off + n]
            big = n > 9000 and bool(((torch.floor(L / rl) >= 3) | (self.per == 0)).all())
            lists.append((_cell_pairs if big else _all_pairs)(y, L, self.per, rl) + off)
            off += n
        self.i, self.j = torch.cat(lists, 1)
        d = x[self.j] - x[self.i]
        L = self.boxes[self.sys[self.i]]
        self.shift = L * torch.round(d / L) * self.per
        if self.pot == "si":   # neighbour table of both directions
            a, b = torch.cat([self.i, self.j]), torch.cat([self.j, self.i])
            sh = torch.cat([self.shift, -self.shift])
            o = torch.argsort(a, stable=True)
            a, b, sh = a[o], b[o], sh[o]
            count = torch.bincount(a, minlength=len(x))
            m = int(count.max())
            slot = torch.arange(len(a), device="cuda") - (torch.cumsum(count, 0) - count)[a]
            self.nb = torch.zeros((len(x), m), dtype=torch.long, device="cuda")
            self.nb_shift = torch.full((len(x), m, 3), 1e3, device="cuda", dtype=F64)
            self.nb[a, slot], self.nb_shift[a, slot] = b, sh

    def atom_energy(self, x):
        if self.pot == "si":
            return self.sw(x)
        d = x.index_select(0, self.j) - x.index_select(0, self.i) - self.shift
        r2 = (d * d).sum(1)
        e = torch.zeros(len(x), device="cuda", dtype=F64)
        if self.pot == "lj":
            s6 = (LJ["sigma"] ** 2 / r2) ** 3
            c6 = (LJ["sigma"] / self.rc) ** 6
            pair = torch.where(r2 < self.rc ** 2, 4 * LJ["eps"] * (s6 * s6 - s6 - c6 * c6 + c6), 0.0)
            return e.index_add(0, self.i, pair)
        A, xi, p, q = self.theta
        r = torch.sqrt(r2)
        t = ((r - CU["rs"]) / (CU["rc"] - CU["rs"])).clamp(0.0, 1.0)
        S = 1 - t ** 3 * (10 - 15 * t + 6 * t * t)
        s = r / CU["r0"] - 1
        g = xi ** 2 * torch.exp(-2 * q * s) * S
        rho = e.index_add(0, self.i, g).index_add(0, self.j, g)
        return e.index_add(0, self.i, 2 * A * torch.exp(-p * s) * S) - torch.sqrt(rho)

    def sw(self, x):
        k = SI
        d = x.index_select(0, self.nb.reshape(-1)).reshape(*self.nb.shape, 3) - x[:, None] - self.nb_shift
        r2 = (d * d).sum(-1)
        on = r2 < self.rc ** 2 * (1 - 1e-9)
        r = torch.sqrt(torch.where(on, r2, 1.0))
        cut = torch.where(on, r - self.rc, -1.0)
        sr = k["sigma"] / r
        pair = k["sw_A"] * k["eps"] * (k["sw_B"] * sr ** 4 - 1.0) * torch.exp(k["sigma"] / cut)
        e = 0.5 * torch.where(on, pair, 0.0).sum(1)
        w = torch.where(on, torch.exp(k["sw_gamma"] * k["sigma"] / cut), 0.0)
        u = torch.where(on[..., None], d, 0.0) / r[..., None]
        c = u @ u.transpose(1, 2)
        h = (c + 1.0 / 3.0) ** 2 * w[:, :, None] * w[:, None, :]
        return e + k["sw_lambda"] * k["eps"] * 0.5 * (h.sum((1, 2)) - h.diagonal(dim1=1, dim2=2).sum(1))

    def total(self, v):
        """Per-system sums of a per-atom vector."""
        if self.S == 1:
            return v.sum().reshape(1)
        return torch.stack([p.sum() for p in torch.split(v, self.counts)])

    def largest(self, v):
        if self.S == 1:
            return v.max().reshape(1)
        return torch.stack([p.max() for p in torch.split(v, self.counts)])

    def energy_forces(self, x):
        self.relist(x)
        x = x.detach().requires_grad_(True)
        e = self.atom_energy(x)
        (f,) = torch.autograd.grad(e.sum(), x)
        return e.detach(), -f


def _fire(x, force, model, mass, dt0, ftol, maxiter):
    """FIRE 2.0 with semi-implicit Euler steps and the default parameters, one
    set of scalars per system; force(x) -> (result, F).  Returns x and the
    last result."""
    S, sys = model.S, model.sys
    v = torch.zeros_like(x)
    dt = torch.full((S,), dt0, device="cuda", dtype=F64)
    alpha = torch.full((S,), 0.25, device="cuda", dtype=F64)
    npos = torch.zeros(S, device="cuda")
    i = torch.zeros(S, device="cuda")

    def each(a):   # a per-system value for every atom
        return a if S == 1 else a[sys][:, None]

    while True:
        res, F = force(x)
        f2a = (F * F).sum(1)
        P, F2 = model.total((F * v).sum(1)), model.total(f2a)
        go = (torch.sqrt(model.largest(f2a)) >= ftol) & (i < maxiter)
        if not bool(go.any()):
            return x, res
        i = i + 1
        up = P > 0
        npos = torch.where(up, npos + 1, 0.0)
        grow = up & (npos > 20)
        dt = torch.where(grow, torch.clamp(dt * 1.1, max=10 * dt0), dt)
        alpha = torch.where(grow, alpha * 0.99, alpha)
        cut = ~up & (i >= 20)
        dt = torch.where(cut & (dt * 0.5 >= 0.02 * dt0), dt * 0.5, dt)
        alpha = torch.where(cut, 0.25, alpha)
        xn = torch.where(each(up), x, x - 0.5 * each(dt) * v)
        vn = torch.where(each(up), v, 0.0) + each(dt / mass) * F
        scale = torch.sqrt(model.total((vn * vn).sum(1)) / F2)
        vn = torch.where(each(up), each(1 - alpha) * vn + each(alpha * scale) * F, vn)
        xn = xn + each(dt) * vn
        x, v = torch.where(each(go), xn, x), torch.where(each(go), vn, v)


def _neb_force(model, ends, L, n_img, k_spring=1.0):
    """Improved-tangent band forces with a climbing image of the packed movable images."""
    e_end = []
    for p in ends:
        m = _Model("cu", p, [L.tolist()], [len(p)], (1, 1, 1))
        e_end.append(m.energy_forces(p)[0].sum())

    def force(x):
        e, F = model.energy_forces(x)
        E = torch.cat([e_end[0].reshape(1), model.total(e), e_end[1].reshape(1)])
        path = torch.cat([ends[0][None], x.reshape(n_img, -1, 3), ends[1][None]])
        d = path[1:] - path[:-1]
        d = d - L * torch.round(d / L)
        tm, tp, F = d[:-1], d[1:], F.reshape(n_img, -1, 3).clone()
        climber = 1 + int(torch.argmax(E[1:-1]))
        for a in range(n_img):
            up, dn = float(E[a + 2] - E[a + 1]), float(E[a + 1] - E[a])
            if up > 0 and dn > 0:
                t = tp[a]
            elif up < 0 and dn < 0:
                t = tm[a]
            else:
                hi, lo = max(abs(up), abs(dn)), min(abs(up), abs(dn))
                t = hi * tp[a] + lo * tm[a] if E[a + 2] > E[a] else lo * tp[a] + hi * tm[a]
            t = t / t.norm()
            along = (F[a] * t).sum()
            spring = k_spring * (tp[a].norm() - tm[a].norm())
            F[a] += t * (-2 * along if a + 1 == climber else spring - along)
        return E, F.reshape(-1, 3)

    return force


def _hessian_times(model, x):
    y = x.detach().requires_grad_(True)
    (g,) = torch.autograd.grad(model.atom_energy(y).sum(), y, create_graph=True)
    return lambda u: torch.autograd.grad((g * u).sum(), y, retain_graph=True)[0]


def exact(case, seed):
    do, pot = case["do"], case.get("pot", "cu")
    mass, dt = _mass_dt(pot)
    cost = work(case)["flops"]
    if cost > 4e11:   # the relaxations of millions of atoms and hundreds of steps
        return None
    if do == "batch":
        x, boxes, counts = _batch(case, seed)
        m = _Model("cu", x, boxes, counts, (1, 1, 1))
        x, e = _fire(x, m.energy_forces, m, mass, dt, case["ftol"], case["maxiter"])
        return {"x": x, "energy": m.total(e).cpu()}
    if do == "neb":
        path, box = _path(case, seed)
        n, M = path.shape[1], case["n_img"]
        L = torch.tensor(box, device="cuda", dtype=F64)
        m = _Model("cu", path[1:-1].reshape(-1, 3), [box] * M, [n] * M, (1, 1, 1))
        band = _Model.__new__(_Model)   # all images are one system for FIRE
        band.S, band.sys = 1, None
        x, E = _fire(path[1:-1].reshape(-1, 3), _neb_force(m, (path[0], path[-1]), L, M), band, mass, dt,
                     case["ftol"], case["maxiter"])
        return {"x": torch.cat([path[:1], x.reshape(M, n, 3), path[-1:]]), "energy": E.cpu().numpy()}
    x, box, periodic, sites, vacant = _system(case, seed)
    m = _Model(pot, x, [box], [len(x)], periodic)
    if do == "relax":
        x, e = _fire(x, m.energy_forces, m, mass, dt, case["ftol"], case["maxiter"])
        return {"x": x, "energy": float(e.sum())}
    if do in ("eval", "noalloc"):
        e, f = m.energy_forces(x)
        return {"forces": f, "energy": e.sum().reshape(1)}
    if do == "energy_grad":
        m.theta.requires_grad_(True)
        y = x.clone().requires_grad_(True)
        e = m.atom_energy(y).sum()
        g, th = torch.autograd.grad(e, [y, m.theta])
        return {"forces": -g, "energy": float(e), "theta": th.cpu().numpy()}
    if do == "hvp":
        u = torch.randn(x.shape, generator=_gen(seed + 1), device="cuda", dtype=F64)
        return {"hu": _hessian_times(m, x)(u)}
    # H lambda = dL/dx with the translations projected out, then lambda . dF/dtheta
    H = _hessian_times(m, x)
    r = _loss_gradient(x, sites, vacant, box)
    r = r - r.mean(0)
    p, lam = r.clone(), torch.zeros_like(r)
    rr = (r * r).sum()
    stop = 1e-24 * rr
    for _ in range(2000):
        if not bool(rr > stop):
            break
        Hp = H(p)
        Hp = Hp - Hp.mean(0)
        a = rr / (p * Hp).sum()
        lam, r = lam + a * p, r - a * Hp
        new = (r * r).sum()
        p, rr = r + (new / rr) * p, new
    m.theta = m.theta.clone().requires_grad_(True)
    y = x.clone().requires_grad_(True)
    (g,) = torch.autograd.grad(m.atom_energy(y).sum(), y, create_graph=True)
    (th,) = torch.autograd.grad(-(g * lam).sum(), m.theta)
    return {"theta": th.cpu().numpy(), "lambda": lam}
