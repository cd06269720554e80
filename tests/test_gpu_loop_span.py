"""The resident kernel leaves for new lists before its barrier's count of arrivals
runs out (2^32, some nine million iterations without a list on 152 blocks); with a
small span it does so every few iterations.  The trajectory does not depend on when
lists are built but for the order of the sums (~1e-15 of the forces): 1e-10 A over 40
iterations, as between the kernel and the chain."""
import numpy as np
import pytest

import fire_inputs as fi
import paper_1908_02038_gb300 as fg

pytestmark = pytest.mark.gpu

CASES = {"rgl": (fi.rgl_vacancy_box(ncell=11, seed=1, n_vac=459, sigma=0.02),
                 fg.Potential(fg.FIRE_POT_RGL, skin=0.3, **fi.RGL_CU), fi.CU_MASS, fi.CU_DT),
         "lj": (fi.lj_fcc_vacancy(seed=1, ncell=7, amp=0.02),
                fg.Potential(fg.FIRE_POT_LJ, skin=0.3, eps=1.0, sigma=1.0, rc_lj=2.5), fi.LJ_MASS,
                fi.LJ_DT)}


@pytest.mark.parametrize("name", CASES)
def test_lists_before_the_count_runs_out(name):
    pytest.importorskip("torch")
    fg.build()
    c, pot, mass, dt = CASES[name]
    got = []
    for span in (None, 1000, 1):   # one list; one every three iterations or so; every iteration
        x = c.x.copy()
        with fg.FireHandle(c.n, mass, pot, dt_start=dt) as h:
            if span:
                fg.fire_diag_set_loop_span(h.h, span)
            r = h.minimize(x, c.box, 1e-12, 40)
            assert fg.fire_diag_resident_loop(h.h) == 1
            for bad in (0, -1, 2 ** 31 + 1):
                with pytest.raises(fg.FireError):
                    fg.fire_diag_set_loop_span(h.h, bad)
        got.append((x, r))
    (x0, r0), (x1, r1), (x2, r2) = got
    assert r0.iterations == r1.iterations == r2.iterations == 40
    assert r0.nbr_builds < r1.nbr_builds and 8 <= r1.nbr_builds <= 21
    assert r2.nbr_builds == 41
    for x, r in got[1:]:
        assert np.abs(x - x0).max() < 1e-10
        assert r.energy == pytest.approx(r0.energy, rel=1e-12)
