"""Captured calls on both sides of the length up to which a survey sorts in one launch: what an earlier, shorter call's
workspace (a quarter larger than asked for) has room for is sorted without allocating."""
import numpy as np
import pytest
import torch

from paper_1204_1225_gb300 import kirchhoff as kh
from paper_1204_1225_gb300 import survey as sv

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("before, now", [(40, 50), (6553, 8191), (6554, 8192), (8193, 10241), (9000, 11250)])
def test_captured_after_a_shorter_call(before, now):
    s = sv.survey_random(np.random.default_rng(now), 3, now, 9, 8, 12, 32, aperture=40.0, n_bins=3, h=10.0)
    d = torch.as_tensor(sv.random_traces(s, 2), device="cuda")
    hdr, fewer = kh.Headers.of(s), kh.Headers.of(s.subset(np.arange(before)))
    plan, other = kh.Plan(s), kh.Plan(s)
    plan.migrate(fewer, d[:before].contiguous())
    got = torch.full(plan.image_shape, float("nan"), device="cuda")
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g):
        plan.migrate(hdr, d, got)
    g.replay()
    plan.sync()
    assert torch.equal(got, other.migrate(hdr, d))
