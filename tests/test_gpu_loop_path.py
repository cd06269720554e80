"""Which path relaxations and evaluations take: the resident kernel at every shape
of its launch that the comparisons with the kernel chain use (they would compare
the chain with itself if it fell back), the chain for what it does not serve."""
import numpy as np
import pytest

import fire_inputs as fi
import paper_1908_02038_gb300 as fg

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    pytest.importorskip("torch")
    fg.build()
    fg.load_library()


def cu(n):
    ncell = 3
    while 4 * ncell ** 3 < n:
        ncell += 1
    return fi.rgl_vacancy_box(ncell=ncell, seed=1, n_vac=4 * ncell ** 3 - n, sigma=0.02)


def rgl(**kw):
    return fg.Potential(fg.FIRE_POT_RGL, skin=0.3, **dict(fi.RGL_CU, **kw))


LJ = fg.Potential(fg.FIRE_POT_LJ, skin=0.3, eps=1.0, sigma=1.0, rc_lj=2.5)


def ran(c, pot, mass=fi.CU_MASS, dt=fi.CU_DT, setup=None, **par):
    """(evaluation, relaxation) in the resident kernel?"""
    with fg.FireHandle(c.n, mass, pot, periodic=c.periodic, dt_start=dt, **par) as h:
        assert fg.fire_diag_resident_loop(h.h) == -1
        if setup:
            setup(h)
        h.energy_forces(c.x, c.box)
        e = fg.fire_diag_resident_loop(h.h)
        h.minimize(c.x.copy(), c.box, 1e-12, 2)
        assert fg.fire_last_error(h.h) == ""
        return e, fg.fire_diag_resident_loop(h.h)


@pytest.mark.parametrize("n", [105, 151, 153, 305, 860, 1216, 1217, 4864, 4865, 17024, 17025, 31680,
                               62499, 65536])
def test_rgl_sizes_run_in_the_resident_kernel(n):
    assert ran(cu(n), rgl()) == (1, 1)


@pytest.mark.parametrize("ncell", [4, 7, 11, 15])
def test_lj_sizes_run_in_the_resident_kernel(ncell):
    assert ran(fi.lj_fcc_vacancy(seed=1, ncell=ncell), LJ, fi.LJ_MASS, fi.LJ_DT) == (1, 1)


def test_slab_runs_in_the_resident_kernel():
    assert ran(fi.rgl_slab(ncell=6, seed=2), rgl()) == (1, 1)


@pytest.mark.parametrize("why", ["size", "newton", "analytic", "fp32", "tiles", "threads", "body",
                                 "chunked", "dmax"])
def test_the_chain_runs_the_rest(why):
    setup = {"tiles": lambda h: h.set_pair_tiles(fg.FIRE_TILES_ON),
             "threads": lambda h: h.set_threads_per_atom(4),
             "body": lambda h: h.set_exec_mode(fg.FIRE_EXEC_GRAPH_WHILE, 8),
             "chunked": lambda h: h.set_exec_mode(fg.FIRE_EXEC_CHUNKED, 4)}.get(why)
    pot = rgl(**{"newton": dict(newton=fg.FIRE_NEWTON_ON),
                 "analytic": dict(pair_eval=fg.FIRE_PAIR_ANALYTIC),
                 "fp32": dict(precision=fg.FIRE_PREC_FP32_PAIR,
                              pair_eval=fg.FIRE_PAIR_ANALYTIC)}.get(why, {}))
    par = dict(dmax=0.1) if why == "dmax" else {}
    assert ran(cu(65537 if why == "size" else 1217), pot, setup=setup, **par) == (0, 0)
