"""The adjoint where a lane or a point is to add nothing: times a hair past the last sample, image values
that are not finite where a trace leaves them out, and depths below the image where v0 + k z is no longer
positive."""
import numpy as np
import pytest

import oracle
from helpers import FP32_REL_L2, gpu_demigrate, rel_l2
from paper_1204_1225_gb300 import survey as sv

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nt", [200, 201, 202, 204, 400])
@pytest.mark.parametrize("past", [0.0, 2.0 ** -11])
def test_time_at_the_last_sample_reaches_no_other(nt, past):
    # one zero-offset trace over column 0 of a constant-velocity line and an image of one point under it,
    # whose two-way time is `past` samples beyond the last one.  Tiles of 32 x 32, two columns of 36 of
    # them in 32 parts: the CTA that meets the point in tile 4 goes on to the shallow tile 36
    v, dt, h = 2000.0, 0.004, 5.0
    nx, nz, jz = 64, 36 * 32, 140
    t0 = 2.0 * jz * h / v - (nt - 1 + past) * dt
    z = np.zeros(1, np.float32)
    s = sv.Survey(dim=2, nx=nx, ny=1, nz=nz, ox=0.0, oy=0.0, oz=0.0, dx=h, dy=h, dz=h, n_bins=1, bin_width=100.0,
                  vel="const", v0=v, k=0.0, weight="one", r0=1000.0, aperture=0.0, nt=nt, t0=t0, dt=dt,
                  sx=z, sy=z, rx=z, ry=z)
    m = np.zeros(s.image_shape, np.float32)
    m[0, 0, 0, jz] = 1.0
    got, _ = gpu_demigrate(s, m)
    assert abs(got[0, -1] - 1.0) < 1e-3
    assert not np.any(got[0, :-1])


def _masked(vel, aperture, nt=220):
    rng = np.random.default_rng(9)
    s = sv.survey_random(rng, 3, 200, 26, 19, 21, nt, vel=vel, weight="one", aperture=aperture, n_bins=2, h=12.5,
                         v0=1700.0, k=0.5 if vel == "linear" else 0.0)
    # shots of 40 receivers: warps of one, two and more source positions
    pick = np.repeat(rng.permutation(s.ntr)[:5], 40)
    s = s.replace(sx=s.sx[pick], sy=s.sy[pick])
    off = np.hypot(s.sx.astype(np.float64) - s.rx, s.sy.astype(np.float64) - s.ry)
    return s.replace(bin_width=(float(off.max()) * 1.0001 + 1.0) / s.n_bins)


@pytest.mark.parametrize("vel", ["const", "linear"])
@pytest.mark.parametrize("aperture, taper", [(0.0, 0.0), (90.0, 0.0), (90.0, 0.4)])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_a_value_that_is_not_finite_stays_with_its_traces(vel, aperture, taper, value):
    s = _masked(vel, aperture).replace(taper=taper)
    m = sv.random_image(s, 3)
    for p in ((0, 7, 11, 9), (1, 18, 25, 20), (0, 0, 0, 0)):
        bad, base, unit = m.copy(), m.copy(), np.zeros_like(m)
        bad[p], base[p], unit[p] = value, 0.0, 1.0
        want, p1 = gpu_demigrate(s, base)
        got, _ = gpu_demigrate(s, bad, plan=p1)
        seen, _ = gpu_demigrate(s, unit, plan=p1)
        hit = seen != 0.0   # samples the point adds to, and their neighbours (a weight of 0 there)
        hit[:, 1:] |= seen[:, :-1] != 0.0
        hit[:, :-1] |= seen[:, 1:] != 0.0
        assert np.array_equal(got[~hit], want[~hit])
        assert not np.all(np.isfinite(got[seen != 0.0])) or not np.any(seen)


@pytest.mark.parametrize("weight", ["one", "obliq"])
@pytest.mark.parametrize("v0", [300.0, 311.0])
def test_depths_below_the_image_with_no_velocity(weight, v0):
    # the image's last depth is the first of 32 in its tile, and v0 + k z reaches zero further down in it
    dz, k, nz = 10.0, -0.5, 33
    assert v0 + k * (nz - 1) * dz > 100.0 > 0.0 > v0 + k * 63 * dz
    s = sv.survey_random(np.random.default_rng(7), 2, 70, 40, 1, nz, 300, vel="linear", weight=weight, n_bins=1, h=1.25,
                         dt=0.05, v0=v0, k=k)
    s = s.replace(dz=dz)
    m = sv.random_image(s, 4)
    got, _ = gpu_demigrate(s, m)
    assert np.any(got)
    # but for the two samples at each edge: a time within 2^-10 samples beyond it counts for the kernel alone
    assert rel_l2(got[:, 2:-2], oracle.demigrate(s, m)[:, 2:-2]) < FP32_REL_L2
