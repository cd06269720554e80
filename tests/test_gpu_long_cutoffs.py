"""The FP64 table form where components of pair separations exceed 8 units of length
(long cut-offs, lengths in bohr or smaller units): positions take a coarser fixed point
there, so that separations still split exactly into two floats.  Every path against
the oracle; forces within ten times the 3.4e-13 (relative to the largest) that cut-offs
up to 8 A give, energies 1e-12; narrow tapers, from the tables' rows and beyond them,
with the bound of test_pair_table_tapers, and a pair closer than r0 / 2 as well."""
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


def scaled(s, ncell=6, **kw):
    P = dict(fi.RGL_CU, **kw)
    c = fi.rgl_vacancy_box(ncell=ncell, seed=4, n_vac=5, sigma=0.04)
    return c.x * s, c.box * s, dict(P, r0=P["r0"] * s, rs=P["rs"] * s, rc=P["rc"] * s), 0.3 * s


SETS = {"rc8": scaled(1.0, 7, rs=7.5, rc=8.0), "rc9": scaled(1.0, 7, rs=8.5, rc=9.0),
        "bohr": scaled(1.8897), "three": scaled(3.0), "ten": scaled(10.0), "ten_rc9": scaled(10.0, 7, rs=8.5, rc=9.0)}


def evaluate(path, x, box, P, skin):
    kw = dict(P, skin=skin, newton=fg.FIRE_NEWTON_OFF if path == "full" else fg.FIRE_NEWTON_AUTO)
    pot = fg.Potential(fg.FIRE_POT_RGL, **kw)
    if path == "batch":
        with fg.FireBatch([len(x)], fi.CU_MASS, pot, dt_start=fi.CU_DT) as h:
            r, f = h.minimize(x.copy(), [box], 1e6, 0, want_forces=True)
        return r[0].energy, f
    with fg.FireHandle(len(x), fi.CU_MASS, pot, dt_start=fi.CU_DT) as h:
        if path in ("chain", "tiles"):
            h.set_exec_mode(fg.FIRE_EXEC_GRAPH_WHILE, 8)
        if path == "tiles":
            h.set_pair_tiles(fg.FIRE_TILES_ON)
        return h.energy_forces(x, box)


@pytest.mark.parametrize("path", ["loop", "chain", "full", "batch"])
@pytest.mark.parametrize("name", SETS)
def test_energies_and_forces(name, path):
    x, box, P, skin = SETS[name]
    eo, fo = oracle.energy_forces(x, box, oracle.Potential("rgl", **P))
    e, f = evaluate(path, x, box, P, skin)
    assert e == pytest.approx(eo, rel=1e-12)
    assert np.abs(f - fo).max() <= 3.4e-12 * np.abs(fo).max()


@pytest.mark.parametrize("name", SETS)
def test_tiles(name):
    """Their neighbour terms are summed in fixed point: the repository's bars."""
    x, box, P, skin = SETS[name]
    eo, fo = oracle.energy_forces(x, box, oracle.Potential("rgl", **P))
    e, f = evaluate("tiles", x, box, P, skin)
    assert e == pytest.approx(eo, rel=1e-12)
    assert np.abs(f - fo).max() <= 1e-10 * np.abs(fo).max()


@pytest.mark.parametrize("path", ["loop", "chain", "full", "tiles", "batch"])
@pytest.mark.parametrize("what", ["taper_rows", "taper", "close"])
def test_narrow_tapers_and_close_pairs(what, path):
    x, box, P, skin = SETS["ten"]
    if what == "taper_rows":     # 0.4 A^2, 26 intervals of 1/64
        P = dict(P, rs=P["rc"] - 0.004, rc=P["rc"])
        tol = 1e-9 * 0.008 / 0.004   # the bound of test_pair_table_tapers at 0.008
    elif what == "taper":        # 0.08 A^2, five intervals: analytic
        P = dict(P, rs=P["rc"] - 0.0008, rc=P["rc"])
        tol = 1e-9 * 10 * 0.008 / 0.0008   # and separations of ten times the size
    else:
        x = x.copy()
        x[1] = x[0] + np.array([0.45 * P["r0"], 0.0, 0.0])
        tol = 1e-10
    eo, fo = oracle.energy_forces(x, box, oracle.Potential("rgl", **P))
    e, f = evaluate(path, x, box, P, skin)
    assert e == pytest.approx(eo, rel=1e-11)
    assert np.abs(f - fo).max() <= tol * np.abs(fo).max()


def test_relaxation():
    x, box, P, skin = SETS["three"]
    dt = 3 * fi.CU_DT   # forces are three times smaller, lengths larger
    xo, ro, _ = oracle.fire2(x, box, oracle.Potential("rgl", **P), oracle.Params(dt_start=dt),
                             fi.CU_MASS, 1e-12, 20)
    y = x.copy()
    with fg.FireHandle(len(x), fi.CU_MASS, fg.Potential(fg.FIRE_POT_RGL, skin=skin, **P),
                       dt_start=dt) as h:
        r = h.minimize(y, box, 1e-12, 20)
    assert r.iterations == ro.iterations == 20
    assert np.abs(y - xo).max() < 1e-9
    assert r.energy == pytest.approx(ro.energy, rel=1e-11)
