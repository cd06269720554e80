"""The FP64 form's pair tables (host copy of what the kernels read) at their
interval edges, for parameter sets that move rs and rc against the intervals.

Intervals are a power of two wide in r^2, h <= r0^2 / 326; the economised
quartic of a function of logarithmic slope a in r^2 is off by (a h / 2)^5 /
1920.  The steepest case is phi at r0 / 2, a = p / r0^2: with p <= 14 and the
first derivative (slope grows by less than 2 there) that is
(14 / 652)^5 * 2^5 / 1920 < 8e-11 of the largest value in the range tested;
above 0.85 r0 (a smaller by 1.7, values by e^-7) it is below 2^-43, the
double-float arithmetic's own error of a few parts."""
import numpy as np
import pytest

import paper_1908_02038_gb300 as fg

CU = dict(A=0.0855, xi=1.224, p=10.96, q=2.278, r0=2.556, rs=4.5, rc=5.0)
SETS = {
    "cu": CU,                                        # rs^2 on an interval edge
    "odd_radii": dict(CU, rs=4.51234, rc=5.43),      # rs^2, rc^2 inside intervals
    "steep": dict(CU, p=14.0, q=3.5),
    "short": dict(CU, rs=1.1, rc=1.9),               # the taper starts below r0 / 2
    "nanometres": dict(A=0.2, xi=2.0, p=10.0, q=3.0, r0=0.2884, rs=0.45, rc=0.56),
}


def reference(P, r):
    r = r.astype(np.longdouble)
    w = np.longdouble(P["rc"]) - np.longdouble(P["rs"])
    t = np.clip((r - np.longdouble(P["rs"])) / w, 0, 1)
    S = 1 - 10 * t ** 3 + 15 * t ** 4 - 6 * t ** 5
    dS = (-30 * t ** 2 + 60 * t ** 3 - 30 * t ** 4) / w
    s = r / np.longdouble(P["r0"]) - 1
    a, b = np.longdouble(P["p"]) / P["r0"], 2 * np.longdouble(P["q"]) / P["r0"]
    phi, g = P["A"] * np.exp(-P["p"] * s), P["xi"] ** 2 * np.exp(-2 * P["q"] * s)
    return np.stack([phi * S, g * S, phi * (-a * S + dS), g * (-b * S + dS)], 1)


@pytest.mark.parametrize("name", SETS)
def test_tables_at_interval_edges(name):
    P = SETS[name]
    h = 2.0 ** np.floor(np.log2(P["r0"] ** 2 / 326.0))
    j = np.arange(int(0.25 * P["r0"] ** 2 / h), int(P["rc"] ** 2 / h) + 2)
    edge = np.concatenate([j * h, (j + 0.5) * h, [P["rs"] ** 2, P["rc"] ** 2]])
    r2 = np.concatenate([edge, edge * (1 - 2e-16), edge * (1 + 2e-16), edge * (1 - 1e-7),
                         edge * (1 + 1e-7)])
    r = np.sqrt(r2)
    r = r[(r > 0.45 * P["r0"]) & (r < P["rc"])]
    tab = fg.fire_diag_rgl_table(fg.Potential(fg.FIRE_POT_RGL, **P).c(), r)
    ref = reference(P, r)
    near = r > 0.85 * P["r0"]
    for k in range(4):
        err = np.abs(tab[:, k] - ref[:, k])
        assert err.max() <= 8e-11 * np.abs(ref[:, k]).max(), k
        if near.any():
            assert err[near].max() <= 4 * 2.0 ** -43 * np.abs(ref[near, k]).max(), k
