"""The resident loop (fire2_loop.cuh) against the kernel chain at the sizes where
its launch changes shape: fewer atoms than SMs, shares of 8 / 9, 32 / 33 and
112 / 113 atoms per block on 152 SMs (lanes per atom 32, 16, 8, 4), LJ and RGL,
every integrator and variant, frozen components, open axes, list rebuilds.
fire_set_exec_mode with a loop-body size selects the chain.

Both follow the same trajectory; they differ in the rounding of the sums
(~1e-15 of the forces), which 40 to 60 iterations of a stable minimisation
carry no further than 1e-10 A (the chain's own runs differ by 1e-12); energies
agree to 1e-12 relative, iteration counts exactly."""
import numpy as np
import pytest

import fire_inputs as fi
import paper_1908_02038_gb300 as fg

pytestmark = pytest.mark.gpu

LJ = dict(eps=1.0, sigma=1.0, rc_lj=2.5)


@pytest.fixture(scope="module", autouse=True)
def lib():
    pytest.importorskip("torch")
    fg.build()
    fg.load_library()


def both(c, pot, mass, dt, maxiter, mask=None, ftol=1e-12, **par):
    out = []
    for chain in (False, True):
        x = c.x.copy()
        with fg.FireHandle(c.n, mass, pot, periodic=c.periodic, dt_start=dt, **par) as h:
            if chain:
                h.set_exec_mode(fg.FIRE_EXEC_GRAPH_WHILE, 8)
            if mask is not None:
                h.set_dof_mask(mask)
            out.append((x, h.minimize(x, c.box, ftol, maxiter)))
    (x0, r0), (x1, r1) = out
    assert (r0.iterations, r0.force_evals, r0.nbr_builds, r0.stop) == \
        (r1.iterations, r1.force_evals, r1.nbr_builds, r1.stop)
    assert np.abs(x0 - x1).max() < 1e-10
    assert r0.energy == pytest.approx(r1.energy, rel=1e-12)
    assert r0.f2norm == pytest.approx(r1.f2norm, rel=1e-6)
    return x0, r0


def cu(n, seed=1, sigma=0.05):
    ncell = 3
    while 4 * ncell ** 3 < n:
        ncell += 1
    return fi.rgl_vacancy_box(ncell=ncell, seed=seed, n_vac=4 * ncell ** 3 - n, sigma=sigma)


RGL = fg.Potential(fg.FIRE_POT_RGL, skin=0.3, **fi.RGL_CU)


@pytest.mark.parametrize("n", [105, 151, 153, 305, 1216, 1217, 4864, 4865, 17024, 17025, 31680])
def test_rgl_sizes(n):
    both(cu(n), RGL, fi.CU_MASS, fi.CU_DT, 40)


@pytest.mark.parametrize("ncell", [4, 7, 11, 15])
def test_lj_sizes(ncell):
    c = fi.lj_fcc_vacancy(seed=ncell, ncell=ncell)
    both(c, fg.Potential(fg.FIRE_POT_LJ, skin=0.3, **LJ), fi.LJ_MASS, fi.LJ_DT, 60)


@pytest.mark.parametrize("integrator", [fg.FIRE_INT_EULER_IMPLICIT, fg.FIRE_INT_EULER_EXPLICIT,
                                        fg.FIRE_INT_VERLET, fg.FIRE_INT_LEAPFROG])
@pytest.mark.parametrize("variant", [fg.FIRE_VARIANT_FIRE2, fg.FIRE_VARIANT_FIRE1])
def test_integrators(integrator, variant):
    both(cu(860, seed=5), RGL, fi.CU_MASS, fi.CU_DT, 50, integrator=integrator, variant=variant)


def test_rebuilds_and_stops():
    c = cu(500, seed=9, sigma=0.25)                    # several lists on the way
    _, r = both(c, RGL, fi.CU_MASS, fi.CU_DT, 60)
    assert r.nbr_builds > 2
    both(c, RGL, fi.CU_MASS, fi.CU_DT, 0)
    _, r = both(cu(500, seed=9), RGL, fi.CU_MASS, fi.CU_DT, 400, ftol=1e-2)
    assert r.stop == fg.FIRE_STOP_FTOL
    _, r = both(cu(500, seed=9), RGL, fi.CU_MASS, fi.CU_DT, 400, vdfmax=0)   # P = 0 at the start
    assert r.stop == fg.FIRE_STOP_MAXVDOTF


def test_frozen_and_open():
    c = fi.rgl_slab(ncell=6, seed=2)
    mask = np.where(c.x[:, 2] < 4.0, 7, 0).astype(np.uint8)
    mask[::7] |= 2
    x, _ = both(c, RGL, fi.CU_MASS, fi.CU_DT, 50, mask=mask)
    for d in range(3):
        sel = (mask >> d) & 1 == 1
        assert np.array_equal(x[sel, d], c.x[sel, d])


def test_time_budget_ends_the_loop():
    c = cu(4865, seed=3)
    with fg.FireHandle(c.n, fi.CU_MASS, RGL, dt_start=fi.CU_DT) as h:
        h.set_time_budget(1e-6)
        with pytest.raises(fg.FireError) as e:
            h.minimize(c.x.copy(), c.box, 1e-12, 100000)
        assert e.value.status == fg.FIRE_ERR_TIMEOUT
        h.set_time_budget(100.0)
        assert h.minimize(c.x.copy(), c.box, 1e-3, 1000).stop == fg.FIRE_STOP_FTOL
