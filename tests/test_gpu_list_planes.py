"""Neighbour lists of atoms in common planes: on a lattice without displacements
half of a half list's candidates lie in the atom's own plane, where the choice
between i -> j and j -> i falls to the second and third components; the queue of
accepted candidates holds them until it decides.  Crowded stencils (several
stagings), a skin of more pairs than the buffer holds, an open axis.  Against
the FP64 oracle at the repository's parity bars (1e-10 relative force, 1e-12
energy; FP32-pair 3e-6 eV/A)."""
import numpy as np
import pytest

import fire_inputs as fi
import oracle
import paper_1908_02038_gb300 as fg

pytestmark = pytest.mark.gpu

OPOT = oracle.Potential("rgl", **fi.RGL_CU)
FORMS = {
    "half": dict(newton=fg.FIRE_NEWTON_ON),
    "full": dict(newton=fg.FIRE_NEWTON_OFF),
    "fp32": dict(precision=fg.FIRE_PREC_FP32_PAIR, pair_eval=fg.FIRE_PAIR_ANALYTIC),
}


@pytest.fixture(scope="module", autouse=True)
def lib():
    pytest.importorskip("torch")
    fg.build()
    fg.load_library()


@pytest.mark.parametrize("form", FORMS)
@pytest.mark.parametrize("ncell,skin,periodic", [(3, 0.3, (1, 1, 1)), (5, 0.3, (1, 1, 1)),
                                                 (6, 2.4, (1, 1, 1)), (6, 0.3, (1, 1, 0)),
                                                 (12, 0.3, (1, 1, 1)), (14, 0.3, (1, 0, 1))])
def test_planes(ncell, skin, periodic, form):
    c = fi.rgl_vacancy_box(ncell=ncell, seed=ncell, n_vac=3, sigma=0.0)
    pot = fg.Potential(fg.FIRE_POT_RGL, skin=skin, **FORMS[form], **fi.RGL_CU)
    with fg.FireHandle(c.n, fi.CU_MASS, pot, periodic=periodic, dt_start=fi.CU_DT) as h:
        e, f = h.energy_forces(c.x, c.box)
    eo, fo = oracle.energy_forces(c.x, c.box, OPOT, periodic=periodic)
    if form == "fp32":
        assert np.abs(f - fo).max() < 3e-6
    else:
        assert np.abs(f - fo).max() <= 1e-10 * np.abs(fo).max()
        assert e == pytest.approx(eo, rel=1e-12)
