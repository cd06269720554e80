"""Stillinger-Weber at other values of gamma than the published 1.2, up to where the
three-body exponential is nothing long before the pair one: energy and forces against
the oracle, with the bounds of the published set."""
import numpy as np
import pytest

import fire_inputs as fi
import oracle
import paper_1908_02038_gb300 as fg

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("gamma", [0.0, 1e-3, 0.5, 1.2, 5.0, 26.0, 40.0, 60.0, 300.0, 1e4])
def test_gamma(gamma):
    pytest.importorskip("torch")
    fg.build()
    oracle.build()
    P = dict(fi.SW_SI, sw_gamma=gamma)
    c = fi.sw_si_vacancy_box(ncell=4, seed=3, n_vac=2, sigma=0.1)
    # second neighbours (3.84 A) spread over the cut-off (3.77 A): pairs up to it
    eo, fo = oracle.energy_forces(c.x, c.box, oracle.Potential("sw", **P), mode=oracle.FORCE_CELLS)
    with fg.FireHandle(c.n, fi.SI_MASS, fg.Potential(fg.FIRE_POT_SW, skin=0.3, **P),
                       dt_start=fi.SI_DT) as h:
        e, f = h.energy_forces(c.x, c.box)
    assert np.abs(f - fo).max() / np.abs(fo).max() < 1e-10
    assert e == pytest.approx(eo, rel=1e-12)


def test_pair_at_the_cutoff():
    """Two atoms from just inside to exactly at the cut-off: the pair energy falls
    to nothing, at gamma = 60 too (it stopped at e^-10 of its scale)."""
    pytest.importorskip("torch")
    fg.build()
    rc = fi.SW_SI["sw_a"] * fi.SW_SI["sigma"]
    pot = fg.Potential(fg.FIRE_POT_SW, skin=0.3, **dict(fi.SW_SI, sw_gamma=60.0))
    with fg.FireHandle(2, fi.SI_MASS, pot, dt_start=fi.SI_DT, periodic=(0, 0, 0)) as h:
        for gap in (1e-2, 1e-6, 1e-13, 0.0):
            x = np.array([[5.0, 5.0, 5.0], [5.0 + rc - gap, 5.0, 5.0]])
            e, f = h.energy_forces(x, [20.0] * 3)
            # A eps (1 - B / a^4) < 15 eV times e^(-sigma / gap)
            assert abs(e) <= 16.0 * np.exp(-fi.SW_SI["sigma"] / max(gap, 1e-3))
            assert np.isfinite(f).all() and np.abs(f).max() <= 1e-60 + (1.0 if gap > 1e-3 else 0.0)
