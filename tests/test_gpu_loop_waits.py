"""A wait of the resident kernel that runs out: the call returns FIRE_ERR_TIMEOUT,
relaxations and evaluations alike, the caller's positions stay as they were, and
the handle works again afterwards.  fire_diag_set_loop_wait(h, 0) lets every wait run
out (after a few hundred polls), whatever has arrived."""
import numpy as np
import pytest

import fire_inputs as fi
import paper_1908_02038_gb300 as fg

pytestmark = pytest.mark.gpu

RGL = fg.Potential(fg.FIRE_POT_RGL, skin=0.3, **fi.RGL_CU)
LJ = fg.Potential(fg.FIRE_POT_LJ, skin=0.3, eps=1.0, sigma=1.0, rc_lj=2.5)
CASES = {"rgl_105": (fi.rgl_vacancy_box(ncell=3, seed=1, n_vac=3, sigma=0.02), RGL),
         "rgl_4865": (fi.rgl_vacancy_box(ncell=11, seed=1, n_vac=459, sigma=0.02), RGL),
         "lj_255": (fi.lj_fcc_vacancy(seed=1, ncell=4), LJ),
         "lj_13499": (fi.lj_fcc_vacancy(seed=1, ncell=15), LJ)}


@pytest.mark.parametrize("name", CASES)
def test_a_wait_that_runs_out(name):
    torch = pytest.importorskip("torch")
    fg.build()
    c, pot = CASES[name]
    mass, dt = (fi.LJ_MASS, fi.LJ_DT) if pot is LJ else (fi.CU_MASS, fi.CU_DT)
    d = torch.from_numpy(c.x).cuda()
    f = torch.empty_like(d)
    e = torch.zeros(1, dtype=torch.float64, device="cuda")
    with fg.FireHandle(c.n, mass, pot, dt_start=dt) as h:
        want = h.energy_forces(c.x, c.box)
        x1 = c.x.copy()
        h.minimize(x1, c.box, 1e-12, 4)
        for _ in range(2):
            fg.fire_diag_set_loop_wait(h.h, 0.0)
            x = c.x.copy()
            for call in (lambda: h.energy_forces(c.x, c.box), lambda: h.minimize(x, c.box, 1e-12, 4),
                         lambda: fg.fire_energy_forces_dev(h.h, d, c.box, f, e),
                         lambda: h.minimize_dev(d, c.box, 1e-12, 4)):
                with pytest.raises(fg.FireError) as err:
                    call()
                assert err.value.status == fg.FIRE_ERR_TIMEOUT and "wait" in str(err.value)
                assert fg.fire_diag_resident_loop(h.h) == 1
            assert np.array_equal(x, c.x) and np.array_equal(d.cpu().numpy(), c.x)
            fg.fire_diag_set_loop_wait(h.h, 5.0)
            got = h.energy_forces(c.x, c.box)
            assert got[0] == want[0] and np.array_equal(got[1], want[1])
            h.minimize(x, c.box, 1e-12, 4)
            assert np.array_equal(x, x1)
        for bad in (-1.0, 61.0, float("nan")):
            with pytest.raises(fg.FireError):
                fg.fire_diag_set_loop_wait(h.h, bad)
