"""The warp-per-atom list build at the shapes where it can go wrong: crowded
cells and stencils (more than a warp, more than the staged candidates), mostly
empty cell grids, few and many cells, more skin pairs than the buffer holds,
atoms one or two boxes away (allowed) and three or very many away (refused).
Forces and energies against the FP64 oracle at the repository's parity bars
(1e-10 relative force, 1e-12 energy; FP32-pair 3e-6 eV/A)."""
import numpy as np
import pytest

import fire_inputs as fi
import oracle
import paper_1908_02038_gb300 as fg

pytestmark = pytest.mark.gpu

OPOT = oracle.Potential("rgl", **fi.RGL_CU)
FORMS = {
    "half": dict(),
    "full": dict(newton=fg.FIRE_NEWTON_OFF),
    "fp32": dict(precision=fg.FIRE_PREC_FP32_PAIR, pair_eval=fg.FIRE_PAIR_ANALYTIC),
}


@pytest.fixture(scope="module", autouse=True)
def lib():
    pytest.importorskip("torch")
    fg.build()
    fg.load_library()


def check(x, box, periodic, form, skin=0.3, xo=None):
    pot = fg.Potential(fg.FIRE_POT_RGL, skin=skin, **FORMS[form], **fi.RGL_CU)
    with fg.FireHandle(len(x), fi.CU_MASS, pot, periodic=periodic, dt_start=fi.CU_DT) as h:
        e, f = h.energy_forces(x, box)
    eo, fo = oracle.energy_forces(x if xo is None else xo, box, OPOT, periodic=periodic)
    if form == "fp32":
        assert np.abs(f - fo).max() < 3e-6
    else:
        assert np.abs(f - fo).max() <= 1e-10 * np.abs(fo).max()
        assert e == pytest.approx(eo, rel=1e-12)


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("shape", ["one_cell", "sparse", "straddling"])
def test_open_boxes(shape, form):
    if shape == "one_cell":     # every atom below the box: one cell, 2,093 candidates
        c = fi.rgl_cluster(radius=18.0, seed=3, centre=(-40.0, -40.0, -40.0), box=60.0)
    elif shape == "sparse":     # 135 atoms in 75^3 cells
        c = fi.rgl_cluster(radius=7.0, seed=4, centre=(200.0, 111.0, 399.0), box=400.0)
    else:
        c = fi.rgl_cluster(radius=12.0, seed=5, centre=(0.0, 15.0, 30.0), box=30.0)
    check(c.x, c.box, (0, 0, 0), form)


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("ncell,skin", [(3, 0.3), (5, 0.3), (5, 1.0), (6, 2.4), (13, 0.3), (14, 0.3)])
def test_periodic_boxes(ncell, skin, form):
    c = fi.rgl_vacancy_box(ncell=ncell, seed=ncell, n_vac=2)
    check(c.x, c.box, (1, 1, 1), form, skin)


@pytest.mark.parametrize("form", FORMS)
def test_atoms_in_other_images(form):
    c = fi.rgl_vacancy_box(ncell=6, seed=8, n_vac=2)
    # one box apart in raw coordinates, two across a face (the image codes' limit)
    k = np.random.default_rng(2).integers(0, 2, size=c.x.shape)
    check(c.x + k * c.box, c.box, (1, 1, 1), form, xo=c.x)


@pytest.mark.parametrize("boxes", [3, 2 ** 18, 2 ** 21, 2 ** 33])
def test_images_too_far_are_refused(boxes):
    c = fi.rgl_vacancy_box(ncell=6, seed=8, n_vac=2)
    x = c.x.copy()
    x[11] += boxes * c.box
    pot = fg.Potential(fg.FIRE_POT_RGL, skin=0.3, **fi.RGL_CU)
    with fg.FireHandle(len(x), fi.CU_MASS, pot, dt_start=fi.CU_DT) as h:
        if boxes < 2 ** 20:
            with pytest.raises(fg.FireError) as e:
                h.energy_forces(x, c.box)
            assert e.value.status == fg.FIRE_ERR_ARG
        else:   # FP32 cannot tell where in the box the atom is: refused or in no pair, never a fault
            try:
                h.energy_forces(x, c.box)
            except fg.FireError as e:
                assert e.status in (fg.FIRE_ERR_ARG, fg.FIRE_ERR_NONFINITE)
