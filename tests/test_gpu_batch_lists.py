"""Batched lists: in-range pairs first, then the skin pairs, of which a thread
holds 24 back; small skins (none or few), ordinary ones and skins of more pairs
than it holds, all-pairs and cell builds, against the oracle.  The tolerances
are the ones of the batched form (FP64 1e-10 of the largest force; FP32 pair
terms 2^-24 x ~50 neighbours x cancellation ~ 1e-5)."""
import numpy as np
import pytest

import fire_inputs as fi
import oracle
import paper_1908_02038_gb300 as fg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    fg.build()
    fg.load_library()


@pytest.mark.parametrize("skin", [0.0, 0.05, 0.3, 1.0, 1.6])
@pytest.mark.parametrize("precision,tol", [(fg.FIRE_PREC_FP64, 1e-10), (fg.FIRE_PREC_FP32_PAIR, 1e-5)])
def test_skins(skin, precision, tol):
    cfgs = fi.rgl_batch(n_sys=5, seed=77, nmin=3, nmax=7)
    x = np.ascontiguousarray(np.concatenate([c.x for c in cfgs]))
    counts = [c.n for c in cfgs]
    pot = fg.Potential(fg.FIRE_POT_RGL, precision=precision, skin=skin, **fi.RGL_CU)
    with fg.FireBatch(counts, fi.CU_MASS, pot, dt_start=fi.CU_DT) as b:
        res, f = b.minimize(x, np.array([c.box for c in cfgs]), 1e-6, 0, want_forces=True)
    off = np.concatenate([[0], np.cumsum(counts)])
    for s, c in enumerate(cfgs):
        eo, fo = oracle.energy_forces(c.x, c.box, oracle.Potential("rgl", **fi.RGL_CU))
        assert np.abs(f[off[s]:off[s + 1]] - fo).max() < tol * np.abs(fo).max(), s
        assert res[s].energy == pytest.approx(eo, rel=tol / 100)
