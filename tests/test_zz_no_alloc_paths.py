"""The kernels that the allocation-free evaluation chooses between: one or four atoms
per warp (from 8,192 atoms on; a last warp with fewer than four), LJ and RGL, table or
library exponentials (from exponents of 600 on), and the accuracy of its forces.

Bars: the FP64 parity bars of the repository (forces 1e-10 relative, energy 1e-12);
the accuracy test's bound lies half-way between how far forces with IEEE square roots
are from a plain 64-bit evaluation, 2.16e-15 +- 0.05e-15 (five seeds, 3,960 and 13,491
atoms), and how far those with r not rounded last were, 2.71e-15."""
import numpy as np
import pytest

import fire_inputs as fi
import oracle
import paper_1908_02038_gb300 as fg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    pytest.importorskip("torch")
    fg.build()
    fg.load_library()
    oracle.build()


def run(c, pot):
    import torch
    d_pos = torch.tensor(c.x, dtype=torch.float64, device="cuda")
    d_f = torch.full_like(d_pos, float("nan"))
    d_e = torch.full((1,), float("nan"), dtype=torch.float64, device="cuda")
    fg.fire_energy_forces_noalloc(pot.c(), d_pos, c.box, c.periodic, d_f, d_e)
    torch.cuda.synchronize()
    return d_f.cpu().numpy(), d_e.item()


def cu(n, **kw):
    ncell = 3
    while 4 * ncell ** 3 < n:
        ncell += 1
    return fi.rgl_vacancy_box(ncell=ncell, seed=3, n_vac=4 * ncell ** 3 - n, sigma=0.06, **kw)


def lj(n):
    c = fi.lj_fcc_vacancy(seed=3, ncell=13, amp=0.05)   # 8,787 atoms
    return fi.Config(c.name, np.ascontiguousarray(c.x[:n]), c.box)


@pytest.mark.parametrize("n", [8191, 8192, 8193, 8194, 8195])
@pytest.mark.parametrize("kind", ["rgl", "lj"])
def test_where_four_atoms_share_a_warp(n, kind):
    if kind == "rgl":
        c, opot = cu(n), oracle.Potential("rgl", **fi.RGL_CU)
        pot = fg.Potential(fg.FIRE_POT_RGL, **fi.RGL_CU)
    else:
        P = dict(eps=1.0, sigma=1.0, rc_lj=2.5)
        c, pot, opot = lj(n), fg.Potential(fg.FIRE_POT_LJ, **P), oracle.Potential("lj", **P)
    f, e = run(c, pot)
    eo, fo = oracle.energy_forces(c.x, c.box, opot, mode=oracle.FORCE_CELLS)
    assert np.abs(f - fo).max() <= 1e-10 * np.abs(fo).max()
    assert e == pytest.approx(eo, rel=1e-12)


@pytest.mark.parametrize("n", [497, 8193])
@pytest.mark.parametrize("pq", [dict(p=650.0, q=2.278), dict(p=599.0, q=2.278), dict(p=10.96, q=310.0)])
def test_steep_exponents(n, pq):
    P = dict(fi.RGL_CU, A=1e-12, **pq)
    c = cu(n)
    f, e = run(c, fg.Potential(fg.FIRE_POT_RGL, **P))
    eo, fo = oracle.energy_forces(c.x, c.box, oracle.Potential("rgl", **P), mode=oracle.FORCE_CELLS)
    assert np.abs(f - fo).max() <= 1e-10 * np.abs(fo).max()
    assert e == pytest.approx(eo, rel=1e-12)


def plain(c, P):
    """Forces by the formulas in 64-bit numpy."""
    idx = []
    for lo in range(0, c.n, 500):
        d = c.x[None] - c.x[lo:lo + 500, None]
        d -= np.round(d / c.box) * c.box
        a, b = np.nonzero((d ** 2).sum(-1) < P["rc"] ** 2)
        idx.append(np.stack([a + lo, b]))
    i, j = np.concatenate(idx, 1)
    i, j = i[i != j], j[i != j]
    d = c.x[j] - c.x[i]
    d -= np.round(d / c.box) * c.box
    r = np.sqrt((d ** 2).sum(1))
    w = P["rc"] - P["rs"]
    t = np.clip((r - P["rs"]) / w, 0, 1)
    S, dS = 1 - t ** 3 * (10 - 15 * t + 6 * t * t), -30 * t * t * (1 - t) ** 2 / w
    s = r / P["r0"] - 1
    phi, g = P["A"] * np.exp(-P["p"] * s), P["xi"] ** 2 * np.exp(-2 * P["q"] * s)
    dphi, dg = phi * (dS - P["p"] / P["r0"] * S), g * (dS - 2 * P["q"] / P["r0"] * S)
    fp = -0.5 / np.sqrt(np.bincount(i, g * S, c.n))
    w = (2 * dphi + (fp[i] + fp[j]) * dg) / r
    return np.stack([np.bincount(i, w * d[:, k], c.n) for k in range(3)], 1)


def test_accuracy_of_forces():
    c = fi.rgl_vacancy_box(ncell=10, seed=1, sigma=0.05)
    f, _ = run(c, fg.Potential(fg.FIRE_POT_RGL, **fi.RGL_CU))
    want = plain(c, fi.RGL_CU)
    assert np.linalg.norm(f - want) < 2.43e-15 * np.linalg.norm(want)
