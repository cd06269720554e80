"""The candidate walk of the allocation-free evaluation at the sizes where it
can go wrong: fewer atoms than a warp, a block or a staged tile, one more and
one fewer, open axes, and raw coordinates several and very many box lengths
outside the box (which the FP32 candidate test must not lose).

Bars: the FP64 parity bars of the repository (forces 1e-10 relative, energy
1e-12); for atoms moved by k box lengths the coordinates themselves lose
k L 2^-53, which the pair stiffness (about 10 forces per Angstrom) carries into
the forces: 1000 boxes of 18 A give 1e-10 relative at most, so 1e-9."""
import numpy as np
import pytest

import fire_inputs as fi
import oracle
import paper_1908_02038_gb300 as fg

pytestmark = pytest.mark.gpu

LJ = dict(eps=1.0, sigma=1.0)


def run(x, box, periodic, pot):
    import torch
    d_pos = torch.tensor(x, dtype=torch.float64, device="cuda")
    d_f = torch.full_like(d_pos, float("nan"))
    d_e = torch.full((1,), float("nan"), dtype=torch.float64, device="cuda")
    fg.fire_energy_forces_noalloc(pot.c(), d_pos, box, periodic, d_f, d_e)
    torch.cuda.synchronize()
    return d_f.cpu().numpy(), d_e.item()


@pytest.fixture(scope="module", autouse=True)
def lib():
    pytest.importorskip("torch")
    fg.build()
    fg.load_library()


@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 31, 33, 64, 65, 255, 256, 257, 459])
@pytest.mark.parametrize("kind", ["rgl", "lj"])
def test_cluster_sizes_on_open_axes(n, kind):
    c = fi.rgl_cluster(radius=10.6, seed=5)
    x = c.x[np.argsort(np.sum((c.x - c.x.mean(0)) ** 2, axis=1))][:n]
    if kind == "rgl":
        pot, opot = fg.Potential(fg.FIRE_POT_RGL, **fi.RGL_CU), oracle.Potential("rgl", **fi.RGL_CU)
    else:
        x = x / 2.3
        pot = fg.Potential(fg.FIRE_POT_LJ, rc_lj=2.5, **LJ)
        opot = oracle.Potential("lj", rc_lj=2.5, **LJ)
    f, e = run(x, c.box, (0, 0, 0), pot)
    eo, fo = oracle.energy_forces(x, c.box, opot, periodic=(0, 0, 0))
    assert np.abs(f - fo).max() <= 1e-10 * max(np.abs(fo).max(), 1e-30)
    assert e == pytest.approx(eo, rel=1e-12, abs=1e-300)


@pytest.mark.parametrize("moved", [3, 5, 1000])
def test_atoms_far_outside_a_periodic_box(moved):
    c = fi.rgl_vacancy_box(ncell=5, seed=41, n_vac=3, sigma=0.08)
    pot = fg.Potential(fg.FIRE_POT_RGL, **fi.RGL_CU)
    f0, e0 = run(c.x, c.box, (1, 1, 1), pot)
    k = np.random.default_rng(1).integers(-moved, moved + 1, size=c.x.shape)
    f, e = run(c.x + k * c.box, c.box, (1, 1, 1), pot)
    assert np.abs(f - f0).max() < 1e-9 * np.abs(f0).max()
    assert e == pytest.approx(e0, rel=1e-9)
