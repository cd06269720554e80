"""A resident loop that cannot be made: the handle takes the kernel chain where the
device does not support it, and reports any other error, after which the next call
makes it.  The failure is a fake of cudaGraphInstantiate in a child process, whose
first call returns the given code without doing anything."""
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
#include <stdlib.h>
int cudaGraphInstantiate(void** exec, void* graph, unsigned long long flags) {
    static int calls = 0;
    static int (*real)(void**, void*, unsigned long long) = 0;
    if (calls++ == 0) return atoi(getenv("FAKE_INSTANTIATE"));
    if (!real) {   /* the library's own runtime, loaded by then */
        void* rt = dlopen("libcudart.so.13", RTLD_LAZY | RTLD_NOLOAD);
        if (!rt) return 999;
        real = (int (*)(void**, void*, unsigned long long))dlsym(rt, "cudaGraphInstantiate");
    }
    return real(exec, graph, flags);
}
"""

CHILD = """
import fire_inputs as fi
import paper_1908_02038_gb300 as fg
c = fi.rgl_vacancy_box(ncell=6, seed=1, n_vac=3)
pot = fg.Potential(fg.FIRE_POT_RGL, skin=0.3, **fi.RGL_CU)
with fg.FireHandle(c.n, fi.CU_MASS, pot, dt_start=fi.CU_DT) as h:
    for _ in range(2):
        try:
            h.minimize(c.x.copy(), c.box, 1e-12, 3)
            print("ok", fg.fire_diag_resident_loop(h.h), repr(fg.fire_last_error(h.h)))
        except fg.FireError as e:
            print("status", e.status)
"""


@pytest.mark.parametrize("code,want", [
    (801, ["ok 0 ''", "ok 0 ''"]),                                   # cudaErrorNotSupported
    (2, ["status %d" % fg.FIRE_ERR_NOMEM, "ok 1 "]),                  # cudaErrorMemoryAllocation
    (999, ["status %d" % fg.FIRE_ERR_CUDA, "ok 1 "]),                 # cudaErrorUnknown
])
def test_what_a_failure_to_make_it_does(tmp_path, code, want):
    fg.build()
    src, lib = tmp_path / "fake.c", tmp_path / "fake.so"
    src.write_text(FAKE)
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", str(lib), str(src), "-ldl"], check=True)
    out = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True,
                         env=dict(os.environ, LD_PRELOAD=str(lib), FAKE_INSTANTIATE=str(code)),
                         timeout=120)
    assert out.returncode == 0, out.stderr
    got = out.stdout.splitlines()
    assert len(got) == 2 and all(g.startswith(w) for g, w in zip(got, want)), got
