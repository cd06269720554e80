"""The resident kernel's line goes by list entries as well as atoms: long cut-offs
take the kernel chain from fewer atoms on."""
import pytest

import fire_inputs as fi
import paper_1908_02038_gb300 as fg

pytestmark = pytest.mark.gpu


def cu(n):
    ncell = 3
    while 4 * ncell ** 3 < n:
        ncell += 1
    return fi.rgl_vacancy_box(ncell=ncell, seed=1, n_vac=4 * ncell ** 3 - n, sigma=0.02)


@pytest.mark.parametrize("kind,n,rc,want", [
    ("rgl", 65536, 5.0, 1), ("rgl", 31680, 8.0, 1), ("rgl", 15900, 10.0, 1), ("rgl", 48000, 10.0, 0),
    ("lj", 15, 2.5, 1), ("lj", 12, 3.5, 1), ("lj", 15, 4.0, 0), ("lj", 7, 5.0, 0)])
def test_line(kind, n, rc, want):
    pytest.importorskip("torch")
    fg.build()
    if kind == "rgl":
        c, mass, dt = cu(n), fi.CU_MASS, fi.CU_DT
        pot = fg.Potential(fg.FIRE_POT_RGL, skin=0.3, **dict(fi.RGL_CU, rs=rc - 0.5, rc=rc))
    else:
        c, mass, dt = fi.lj_fcc_vacancy(seed=1, ncell=n), fi.LJ_MASS, fi.LJ_DT
        pot = fg.Potential(fg.FIRE_POT_LJ, skin=0.3, eps=1.0, sigma=1.0, rc_lj=rc)
    with fg.FireHandle(c.n, mass, pot, dt_start=dt) as h:
        h.energy_forces(c.x, c.box)
        assert fg.fire_diag_resident_loop(h.h) == want
        h.minimize(c.x.copy(), c.box, 1e-12, 2)
        assert fg.fire_diag_resident_loop(h.h) == want
