"""The check of the ln(1 + rho) fits: the reported coefficients, evaluated against log1p at the points of the
check, meet the budget exactly where a fit of that length was accepted, over gradients, spacings and tiles; and
a report does not depend on the reports before it."""
import numpy as np
import pytest

from paper_1204_1225_gb300 import kirchhoff as kh
from paper_1204_1225_gb300 import survey as sv

TILES = [(16, 16, 1), (8, 8, 4), (32, 8, 1)]


def _desc(seed):
    rng = np.random.default_rng(seed)
    s = sv.survey_random(rng, 3, 10, 20, 20, 40, 200, vel="linear", v0=float(rng.uniform(400, 4000)),
                         k=float(10 ** rng.uniform(-4, 0.5)), h=float(rng.uniform(1, 50)))
    return s.replace(dt=float(10 ** rng.uniform(-3, -1.7)))


def _worst(r, c1):
    """Largest |x (1 + x Q) - log1p(x)| of the per-leg fit, Q by FP32 Horner steps for the short lengths."""
    b, n = r["leg_bound"], r["leg_terms"]
    x = np.expm1(-b) + (np.expm1(b) - np.expm1(-b)) * np.arange(4001) / 4000.0
    q = np.asarray(r["coef"], np.float32)[1:n].astype(np.float64) / c1
    if n <= 8:
        x = x.astype(np.float32).astype(np.float64)
    t = x * r["scale"] + r["offset"]
    p = np.zeros_like(x)
    for c in q[::-1]:
        p = p * t + c
    return float(np.max(np.abs(x * (1.0 + x * p) - np.log1p(x))))


@pytest.mark.parametrize("seed", range(24))
def test_accepted_fits_meet_the_budget(seed):
    s = _desc(seed)
    tile = TILES[seed % 3]
    try:
        r = kh.kirchhoff_fit_report(kh.desc_from(s), tile)
    except kh.KirchhoffError as e:
        assert e.status == kh.KH_ERR_UNSUPPORTED
        return
    c1 = 1.0 / (abs(s.k) * s.dt)
    tol = 0.5 * max(5e-6 * abs(s.k) * s.dt, 1e-12)
    # the coefficients are rounded once more by the scaling with C1 (2^-24 of x^2 Q each), and the
    # short lengths' Horner steps round in FP32
    b = r["leg_bound"]
    assert _worst(r, c1) <= tol + 4 * 2.0 ** -24 * np.expm1(b) ** 2


def test_reports_do_not_depend_on_those_before():
    a = {i: repr(kh.kirchhoff_fit_report(kh.desc_from(_desc(i)), (8, 8, 4))) for i in (3, 5)}
    for i in (5, 3, 5, 5, 3):
        assert repr(kh.kirchhoff_fit_report(kh.desc_from(_desc(i)), (8, 8, 4))) == a[i]
