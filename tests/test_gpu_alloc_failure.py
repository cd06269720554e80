"""A device allocation that fails in a call: the call returns FIRE_ERR_NOMEM, and the
next ones on the handle work.  The failure is a fake of cudaMalloc in a child process
that refuses more than a given size."""
import os
import subprocess
import sys

import pytest

import paper_1908_02038_gb300 as fg

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAKE = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stddef.h>
static size_t most = (size_t)-1;
void fake_most(size_t bytes) { most = bytes; }
int cudaMalloc(void** p, size_t bytes) {
    static int (*real)(void**, size_t) = 0;
    if (bytes > most) return 2;   /* cudaErrorMemoryAllocation */
    if (!real) {
        void* rt = dlopen("libcudart.so.13", RTLD_LAZY | RTLD_NOLOAD);
        if (!rt) return 999;
        real = (int (*)(void**, size_t))dlsym(rt, "cudaMalloc");
    }
    return real(p, bytes);
}
"""

CHILD = """
import ctypes, os
import numpy as np
import fire_inputs as fi
import paper_1908_02038_gb300 as fg
most = ctypes.CDLL(os.environ["LD_PRELOAD"]).fake_most
most.argtypes = [ctypes.c_size_t]
ALL = 2 ** 64 - 1

def refused(call):
    try:
        call()
    except fg.FireError as e:
        return e.status == fg.FIRE_ERR_NOMEM
    return False

RGL = fg.Potential(fg.FIRE_POT_RGL, skin=0.3, **fi.RGL_CU)
c = fi.rgl_cluster(radius=10.0)
for chain in (False, True):   # cells: 5^3, then 37^3 and more
    with fg.FireHandle(c.n, fi.CU_MASS, RGL, periodic=(0, 0, 0), dt_start=fi.CU_DT) as h:
        if chain:
            h.set_exec_mode(fg.FIRE_EXEC_GRAPH_WHILE, 8)
        e, f = h.energy_forces(c.x, c.box)
        most(100000)
        assert refused(lambda: h.energy_forces(c.x, [200.0] * 3))
        assert refused(lambda: h.minimize(c.x.copy(), [200.0] * 3, 1e-12, 2))
        e1, f1 = h.energy_forces(c.x, c.box)
        most(ALL)
        e2, f2 = h.energy_forces(c.x, [200.0] * 3)
        for a, b in ((e1, f1), (e2, f2)):
            assert abs(a - e) <= 1e-12 * abs(e) and np.abs(b - f).max() <= 1e-12 * np.abs(f).max()

d = fi.rgl_vacancy_box(ncell=5, seed=1, n_vac=3)   # lists: a denser box needs longer ones
with fg.FireHandle(d.n, fi.CU_MASS, RGL, dt_start=fi.CU_DT) as h:
    e, f = h.energy_forces(d.x, d.box)
    most(50000)
    assert refused(lambda: h.energy_forces(d.x * 0.9, np.array(d.box) * 0.9))
    assert refused(lambda: h.energy_forces(d.x, d.box))   # given up for the longer ones
    most(ALL)
    e1, f1 = h.energy_forces(d.x, d.box)
    assert abs(e1 - e) <= 1e-12 * abs(e) and np.abs(f1 - f).max() <= 1e-12 * np.abs(f).max()

with fg.FireBatch([d.n], fi.CU_MASS, RGL, dt_start=fi.CU_DT) as h:
    x = d.x.copy()
    most(50000)
    assert refused(lambda: h.minimize(d.x.copy(), [list(d.box)], 1e-12, 2))
    most(ALL)
    r, _ = h.minimize(x, [list(d.box)], 1e-12, 2)
    assert r[0].iterations == 2
import torch
th = [fi.RGL_CU[k] for k in ("A", "xi", "p", "q")]
x = torch.from_numpy(d.x).cuda()
with fg.FireHandle(d.n, fi.CU_MASS, RGL, dt_start=fi.CU_DT) as h:
    h.energy_forces(d.x, d.box)
    for bytes in (10000, 20000, 70000):   # the arrays of 16 kB, the vectors, the list
        most(bytes)
        assert refused(lambda: fg.fire_rgl_energy_grad_dev(h.h, x, d.box, th))
    most(ALL)
    e, _ = fg.fire_rgl_energy_grad_dev(h.h, x, d.box, th)
    assert abs(e - e1) <= 1e-12 * abs(e1)
print("done")
"""


def test_calls_after_a_refused_allocation(tmp_path):
    fg.build()
    src, lib = tmp_path / "fake.c", tmp_path / "fake.so"
    src.write_text(FAKE)
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", str(lib), str(src), "-ldl"], check=True)
    out = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True,
                         env=dict(os.environ, LD_PRELOAD=str(lib)), timeout=300)
    assert out.returncode == 0 and out.stdout.splitlines()[-1] == "done", out.stderr
