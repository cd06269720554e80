"""Evaluations of small and mid-size systems run as one launch of the resident
loop: against the kernel chain (fire_set_exec_mode with a loop-body size selects
it) at the sizes where the launch changes shape, through the host and the device
entry point, before and after a relaxation on the same handle.

The two differ in the order of the sums and in half against full lists
(~1e-15 of the terms, of which an atom has ~50): 1e-12 of the largest force
component and 1e-13 of the energy hold with a margin of ten."""
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
    return fi.rgl_vacancy_box(ncell=ncell, seed=3, n_vac=4 * ncell ** 3 - n, sigma=0.08)


RGL = fg.Potential(fg.FIRE_POT_RGL, skin=0.3, **fi.RGL_CU)
LJ = fg.Potential(fg.FIRE_POT_LJ, skin=0.3, eps=1.0, sigma=1.0, rc_lj=2.5)


def close(a, b):
    assert abs(a[0] - b[0]) <= 1e-13 * abs(b[0])
    assert np.abs(a[1] - b[1]).max() <= 1e-12 * np.abs(b[1]).max()


def check(c, pot, mass, dt):
    import torch
    with fg.FireHandle(c.n, mass, pot, periodic=c.periodic, dt_start=dt) as h:
        h.set_exec_mode(fg.FIRE_EXEC_GRAPH_WHILE, 8)
        want = h.energy_forces(c.x, c.box)
    with fg.FireHandle(c.n, mass, pot, periodic=c.periodic, dt_start=dt) as h:
        close(h.energy_forces(c.x, c.box), want)
        close((h.energy_forces(c.x, c.box, want_forces=False)[0], want[1]), want)
        h.minimize(c.x.copy(), c.box, 1e-9, 3)
        d, f = torch.from_numpy(c.x).cuda(), torch.empty(c.n, 3, dtype=torch.float64, device="cuda")
        e = torch.zeros(1, dtype=torch.float64, device="cuda")
        fg.fire_energy_forces_dev(h.h, d, c.box, f, e)
        torch.cuda.synchronize()
        close((e.item(), f.cpu().numpy()), want)


@pytest.mark.parametrize("n", [105, 153, 1217, 4865, 17025, 62499])
def test_rgl(n):
    check(cu(n), RGL, fi.CU_MASS, fi.CU_DT)


def test_open_axis():
    check(fi.rgl_slab(ncell=6, seed=2), RGL, fi.CU_MASS, fi.CU_DT)


@pytest.mark.parametrize("ncell", [4, 15])
def test_lj(ncell):
    check(fi.lj_fcc_vacancy(seed=4, ncell=ncell), LJ, fi.LJ_MASS, fi.LJ_DT)


def test_not_finite_is_reported():
    c = cu(500)
    x = c.x.copy()
    x[1] = x[0]
    with fg.FireHandle(c.n, fi.CU_MASS, RGL, dt_start=fi.CU_DT) as h:
        got = []
        for chain in (False, True):
            if chain:
                h.set_exec_mode(fg.FIRE_EXEC_GRAPH_WHILE, 8)
            try:
                h.energy_forces(x, c.box)
                got.append(None)
            except fg.FireError as e:
                got.append(e.status)
        assert got[0] == got[1]
        h.set_exec_mode(fg.FIRE_EXEC_GRAPH_WHILE, 0)
        h.energy_forces(c.x, c.box)
