"""Gridded-model migration where a warp skips the traces at the end of one ring stage and at the start of
the next: the receiver nodes it read ahead for a skipped trace belong to no other."""
import numpy as np
import pytest

import oracle
from helpers import FP32_REL_L2, gpu_migrate, rel_l2
from paper_1204_1225_gb300 import kirchhoff as kh
from paper_1204_1225_gb300 import survey as sv

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("run", [1, 7, 16, 31, 32, 40, 63])
@pytest.mark.parametrize("m", [2, 4])
def test_traces_skipped_across_stages(run, m):
    # windows so short that a stage holds its 64 traces, and bins so many that the one in use is not cut
    # into parts: midpoints at the left end of a 64-column tile for
    # the first `run` traces of a stage and at the right end for the others, turned about from stage to
    # stage; a warp of 32 columns sees one kind only
    rng = np.random.default_rng(run)
    n = 4 * 64
    i = np.arange(n)
    left = (i % 64 < run) == (i // 64 % 2 == 0)
    mid = np.where(left, 60.0, 570.0) + rng.integers(-6, 7, n) * 5.0
    half = rng.integers(0, 12, n) * 5.0
    f = lambda a: a.astype(np.float32)
    s = sv.survey_random(rng, 2, n, 64, 1, 48, 32, aperture=170.0, n_bins=16, h=10.0, dt=0.08, v0=1800.0, k=0.5)
    s = s.replace(sx=f(mid - half), rx=f(mid + half), bin_width=200.0)
    s = sv.vxz_model(s, m, lens_dv=-400.0, lens_r=150.0)
    d = sv.random_traces(s, 8, smooth=5)
    p = kh.Plan(s)
    p.set_option(kh.KH_OPT_SPATIAL_SORT, 0)
    got, _ = gpu_migrate(s, d, plan=p)
    assert rel_l2(got, oracle.migrate(s, d)) < FP32_REL_L2
