"""A cluster in a large open box: more cells than 32 bits of threads, and than 32 bits
of cells, give the energies and forces of a small box.  The positions are the same but
for the shift, which is a multiple of 2^-8 A on coordinates rounded to 2^-30 A, so that
the FP64 separations are the same numbers; sums in another order differ by 1e-15 of the
terms, of which an atom has ~50: 1e-12 of the largest force, 1e-13 of the energy."""
import numpy as np
import pytest

import fire_inputs as fi
import paper_1908_02038_gb300 as fg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("box", [[2725.0, 2725.0, 2725.0],      # 2^27 cells of 5.3 A at 2,716 A
                                 [9000.0, 9000.0, 9000.0],      # 4.9e9 of them
                                 [30.0, 200000.0, 60000.0]])
@pytest.mark.parametrize("form", ["loop", "chain", "analytic"])
def test_large_open_box(box, form):
    pytest.importorskip("torch")
    fg.build()
    c = fi.rgl_cluster(radius=10.0)
    x = np.round(c.x * 2.0 ** 30) / 2.0 ** 30
    far = x + np.floor(np.array(box) - 30.0)   # the last cells
    pot = fg.Potential(fg.FIRE_POT_RGL, skin=0.3, **fi.RGL_CU,
                       pair_eval=fg.FIRE_PAIR_ANALYTIC if form == "analytic" else fg.FIRE_PAIR_TABLE)
    with fg.FireHandle(c.n, fi.CU_MASS, pot, periodic=(0, 0, 0), dt_start=fi.CU_DT) as h:
        if form == "chain":
            h.set_exec_mode(fg.FIRE_EXEC_GRAPH_WHILE, 8)
        e0, f0 = h.energy_forces(x, c.box)
        e, f = h.energy_forces(far, box)
    assert e == pytest.approx(e0, rel=1e-13)
    assert np.abs(f - f0).max() <= 1e-12 * np.abs(f0).max()
