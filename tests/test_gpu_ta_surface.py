"""True-amplitude weight with sources and receivers on surface columns of the grid, where a leg's
length is 0 and the weight is defined as 0: migration and demigration against the oracle, with
approximate and exact roots, anti-aliasing on and off."""
import numpy as np
import pytest

import oracle
from helpers import FP32_REL_L2, gpu_demigrate, gpu_migrate, rel_l2
from paper_1204_1225_gb300 import survey as sv

pytestmark = pytest.mark.gpu


def _survey(dim, aa):
    rng = np.random.default_rng(17 + dim)
    s = sv.survey_random(rng, dim, 90, 21, 13, 20, 300, weight="ta", n_bins=2, h=12.5, v0=1900.0)

    def snap(a, n):   # onto the grid's columns
        return (np.clip(np.round(a / 12.5), 0, n - 1) * 12.5).astype(np.float32)

    s = s.replace(sx=snap(s.sx, s.nx), rx=snap(s.rx, s.nx), sy=snap(s.sy, s.ny), ry=snap(s.ry, s.ny), aa_spacing=aa)
    same = np.arange(s.ntr) % 9 == 0   # some with source and receiver at one point
    return s.replace(rx=np.where(same, s.sx, s.rx), ry=np.where(same, s.sy, s.ry))


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("fast_math", [True, False])
@pytest.mark.parametrize("aa", [0.0, 25.0])
def test_surface_points_under_sources_and_receivers(dim, fast_math, aa):
    s = _survey(dim, aa)
    d = sv.random_traces(s, 5, smooth=5)
    got, p = gpu_migrate(s, d, fast_math=fast_math)
    assert np.all(got[..., 0] == 0.0)
    assert rel_l2(got, oracle.migrate(s, d)) < FP32_REL_L2
    m = oracle.migrate(s, d).astype(np.float32)
    m[..., 0] = sv.random_image(s, 6)[..., 0]   # what lies on the surface row is given the weight 0
    back, _ = gpu_demigrate(s, m, fast_math=fast_math, plan=p)
    assert rel_l2(back, oracle.demigrate(s, m)) < FP32_REL_L2
