"""Narrow tapers: rows of the pair tables where the taper spans eight intervals
or more, the analytic functions below (rc = 5: 8 h = 1/8 A^2, w = rc - rs = 0.0125).

Host: against the formulas in long double.  Values are off by at most 6 / 512 n^-5
of the untapered function over n >= 6 intervals (the economised quintic), 1.5e-6;
the derivative by the same of (2 / w) f, since S' is a quartic, whose fifth-degree
part comes from the exponential only.  The tests against rs and rc are made in FP32
(r off by 3e-7 at most): 10 (3e-7 / w)^3 and 30 (3e-7 / w)^2 / w more.

Device: separations are good to 2e-13 A, so that a taper's force, S' <= 1.9 / w with
S'' <= 5.8 / w^2, is off by 3 / w times that, 8e-11 of its peak at w = 0.008: 1e-9 of
the largest force, and 1e-11 of the energy (S off by 1.9 / w times that)."""
import numpy as np
import pytest

import fire_inputs as fi
import oracle
import paper_1908_02038_gb300 as fg
from test_pair_tables import CU, reference


@pytest.mark.parametrize("w", [0.05, 0.0126, 0.0125, 0.0095, 0.0093, 4e-3, 1e-3, 1e-4, 1e-5])
def test_narrow_tapers_on_the_host(w):
    P = dict(CU, rs=CU["rc"] - w)
    rng = np.random.default_rng(1)
    r = np.concatenate([rng.uniform(P["rs"], P["rc"], 4000), P["rs"] + w * rng.uniform(-2, 0, 500),
                        rng.uniform(2.0, 5.0, 4000), [P["rs"], np.nextafter(P["rc"], 0)]])
    tab = fg.fire_diag_rgl_table(fg.Potential(fg.FIRE_POT_RGL, **P).c(), r)
    ref, whole = reference(P, r), reference(dict(P, rs=50.0, rc=51.0), r)
    for k in range(2):
        f = whole[:, k]
        at_rc = 3e-7 / w
        assert (np.abs(tab[:, k] - ref[:, k]) <= (1.6e-6 + 10 * at_rc ** 3) * f).all()
        assert (np.abs(tab[:, 2 + k] - ref[:, 2 + k]) <=
                (1.6e-6 * 2 + 30 * at_rc ** 2) / w * f).all()


@pytest.mark.gpu
@pytest.mark.parametrize("path", ["loop", "chain", "full", "tiles", "batch", "confirm"])
def test_narrow_taper_on_the_device(path):
    pytest.importorskip("torch")
    fg.build()
    fg.load_library()
    oracle.build()
    # a fourth of a fourth-shell pair's spread (5.11 A) lies in the taper
    P = dict(fi.RGL_CU, rs=5.107, rc=5.115)
    c = fi.rgl_vacancy_box(ncell=7, seed=4, n_vac=5, sigma=0.01)
    e0, f0 = oracle.energy_forces(c.x, c.box, oracle.Potential("rgl", **P))
    pot = dict(P, skin=0.3, newton=fg.FIRE_NEWTON_OFF if path == "full" else fg.FIRE_NEWTON_AUTO)
    if path == "confirm":   # FP32-pair: the FP64 passes end the relaxation
        pot.update(precision=fg.FIRE_PREC_FP32_PAIR, pair_eval=fg.FIRE_PAIR_ANALYTIC)
    pot = fg.Potential(fg.FIRE_POT_RGL, **pot)
    tol = 1e-9 * np.abs(f0).max()
    if path == "batch":
        with fg.FireBatch([c.n], fi.CU_MASS, pot, dt_start=fi.CU_DT) as h:
            r, f = h.minimize(c.x.copy(), [c.box], 1e3, 0, want_forces=True)
        e = r[0].energy
    elif path == "confirm":
        with fg.FireHandle(c.n, fi.CU_MASS, pot, dt_start=fi.CU_DT) as h:
            r = h.minimize(c.x.copy(), c.box, 1e3, 10)   # stops at once, confirmed
        assert r.iterations == 0 and r.energy == pytest.approx(e0, rel=1e-11)
        assert abs(r.fmax_atom - np.sqrt((f0 ** 2).sum(1).max())) <= 2 * tol
        return
    else:
        with fg.FireHandle(c.n, fi.CU_MASS, pot, dt_start=fi.CU_DT) as h:
            if path in ("chain", "tiles"):
                h.set_exec_mode(fg.FIRE_EXEC_GRAPH_WHILE, 8)
            if path == "tiles":
                h.set_pair_tiles(fg.FIRE_TILES_ON)
            e, f = h.energy_forces(c.x, c.box)
    assert e == pytest.approx(e0, rel=1e-11)
    assert np.abs(f - f0).max() <= tol
