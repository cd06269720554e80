"""Pair tables of the FP64 form (host copy) where lengths are other numbers than in
Angstrom: bohr and beyond, a wide taper's share of a row, an r0 far below rc.

An interval of width h puts a polynomial of a function of logarithmic slope a in
r^2 off by (a h / 2)^5 / 1920.  phi is the steepest, a = p / r0^2 at r0 / 2 and
less than twice that for its derivative: (p h / (2 r0^2))^5 2^5 / 1920 of the largest
value; with h <= r0^2 / 1304 (lengths in bohr or more) that is below 2^-43 for
p <= 14.  The arithmetic adds a few parts of 2^-43: 4 are allowed."""
import time

import numpy as np
import pytest

import paper_1908_02038_gb300 as fg
from test_pair_tables import CU, reference


def lengths(s, **kw):
    P = dict(CU, **kw)
    return dict(P, r0=P["r0"] * s, rs=P["rs"] * s, rc=P["rc"] * s)


SETS = {   # parameters, width of the intervals
    "r0_3.4": (dict(CU, r0=3.4, rs=6.0, rc=6.65), 2.0 ** -6),
    "bohr": (lengths(1.8897), 2.0 ** -6),
    "bohr_steep": (lengths(1.8897, p=14.0, q=3.5), 2.0 ** -6),
    "tens": (lengths(10.0), 2.0 ** -1),
    "hundreds": (lengths(100.0), 2.0 ** 5),
    "tens_narrow_taper": (lengths(10.0, rs=4.95), 2.0 ** -4),
    "r0_far_below_rc": (dict(CU, r0=0.1, p=1.4, q=0.6), 2.0 ** -11),
    "r0_tiny": (dict(CU, r0=0.02, p=0.28, q=0.12), 2.0 ** -11),
    "r0_beyond_rc": (dict(CU, r0=40.0), 2.0 ** -6),
}


@pytest.mark.parametrize("name", SETS)
def test_errors_do_not_depend_on_the_unit_of_length(name):
    P, h = SETS[name]
    rng = np.random.default_rng(2)
    lo = min(0.45 * P["r0"], 0.5 * P["rs"])
    r = np.sqrt(np.concatenate([rng.uniform(lo ** 2, P["rc"] ** 2, 20000),
                                rng.uniform(P["rs"] ** 2, P["rc"] ** 2, 5000),
                                rng.uniform(lo ** 2, min(4 * lo, P["rc"]) ** 2, 5000)]))
    t0 = time.time()
    tab = fg.fire_diag_rgl_table(fg.Potential(fg.FIRE_POT_RGL, **P).c(), r)
    assert time.time() - t0 < 5.0
    ref = reference(P, r)
    bound = (P["p"] * h / (2 * P["r0"] ** 2)) ** 5 * 32 / 1920 + 4 * 2.0 ** -43
    for k in range(4):
        assert np.abs(tab[:, k] - ref[:, k]).max() <= bound * np.abs(ref[:, k]).max(), k
