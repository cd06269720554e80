"""Kernels whose dynamic shared memory depends on the handle: a handle that needs
less must not take the room from one that needs more (the limit is the process's),
in any order and with a thread per handle.  Sizes of one launch shape of the
resident kernel each: 1,217 to 4,864 atoms (16 lanes) and 17,025 to 19,456 (4)."""
import threading

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
    return fi.rgl_vacancy_box(ncell=ncell, seed=2, n_vac=4 * ncell ** 3 - n, sigma=0.03)


RGL = fg.Potential(fg.FIRE_POT_RGL, skin=0.3, **fi.RGL_CU)


@pytest.mark.parametrize("sizes", [(1300, 3960), (3960, 1300), (17025, 19400), (19400, 17025)])
def test_either_order_keeps_the_resident_kernel(sizes):
    for n in sizes + sizes:
        c = cu(n)
        with fg.FireHandle(c.n, fi.CU_MASS, RGL, dt_start=fi.CU_DT) as h:
            h.energy_forces(c.x, c.box)
            assert fg.fire_diag_resident_loop(h.h) == 1
            h.minimize(c.x.copy(), c.box, 1e-12, 3)
            assert fg.fire_diag_resident_loop(h.h) == 1


def test_fp32_tables_of_two_cutoffs():
    c = fi.rgl_vacancy_box(ncell=8, seed=3, n_vac=2, sigma=0.03)
    got = {}
    for rc in (13.0, 5.0):   # 1,400 and 250 rows: 67 and 12 kB
        pot = fg.Potential(fg.FIRE_POT_RGL, skin=0.3, precision=fg.FIRE_PREC_FP32_PAIR,
                           pair_eval=fg.FIRE_PAIR_TABLE, **dict(fi.RGL_CU, rs=rc - 0.5, rc=rc))
        got[rc] = fg.FireHandle(c.n, fi.CU_MASS, pot, dt_start=fi.CU_DT)
    try:
        for rc in (13.0, 5.0, 13.0):
            e, f = got[rc].energy_forces(c.x, c.box)
            assert np.isfinite(e) and np.isfinite(f).all()
    finally:
        for h in got.values():
            h.close()


@pytest.mark.parametrize("sizes", [(1300, 4800), (31000, 19400)])
def test_two_threads(sizes):
    """A handle per thread: no call fails, and every result is what the handle
    gives alone (the resident kernel's results do not depend on timing)."""
    errors = []

    def work(n):
        try:
            c = cu(n)
            with fg.FireHandle(c.n, fi.CU_MASS, RGL, dt_start=fi.CU_DT) as h:
                e0, f0 = h.energy_forces(c.x, c.box)
                x0 = c.x.copy()
                h.minimize(x0, c.box, 1e-12, 5)
                for _ in range(40):
                    e, f = h.energy_forces(c.x, c.box)
                    x = c.x.copy()
                    h.minimize(x, c.box, 1e-12, 5)
                    assert fg.fire_diag_resident_loop(h.h) == 1
                    assert e == e0 and np.array_equal(f, f0) and np.array_equal(x, x0)
        except Exception as e:   # noqa: BLE001 - reported by the test's thread
            errors.append(repr(e))

    threads = [threading.Thread(target=work, args=(n,)) for n in sizes]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors


def test_two_threads_of_batches():
    errors = []

    def work(ncell):
        try:
            cs = [fi.rgl_vacancy_box(ncell=ncell, seed=s, n_vac=1, sigma=0.03) for s in range(3)]
            pos = np.concatenate([c.x for c in cs])
            boxes = [list(c.box) for c in cs]
            with fg.FireBatch([c.n for c in cs], fi.CU_MASS, RGL, dt_start=fi.CU_DT) as h:
                for _ in range(60):
                    h.minimize(pos.copy(), boxes, 1e-12, 1)
        except Exception as e:   # noqa: BLE001
            errors.append(repr(e))

    threads = [threading.Thread(target=work, args=(n,)) for n in (3, 12)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors
