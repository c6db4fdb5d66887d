"""The adjoint where a lane or a point is to add nothing: times a hair past the last sample."""
import numpy as np
import pytest

from helpers import gpu_demigrate
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
