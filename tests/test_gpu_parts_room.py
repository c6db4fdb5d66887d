"""Traces of a bin cut into parts where the partial images cannot be held (a captured call whose workspace
is too small, a batch on a full device): the parts are added in the same order as with them, so the
images are the same bits."""
import numpy as np
import pytest
import torch

from paper_1204_1225_gb300 import kirchhoff as kh
from paper_1204_1225_gb300 import survey as sv

pytestmark = pytest.mark.gpu


def _captured(fn):
    g = torch.cuda.CUDAGraph()
    torch.cuda.synchronize()
    with torch.cuda.graph(g):
        fn()
    g.replay()
    torch.cuda.synchronize()


@pytest.mark.parametrize("vel, weight, dtype", [("const", "ta", torch.float32), ("linear", "obliq", torch.float32),
                                                ("linear", "one", torch.float16), ("pstm", "obliq", torch.float32)])
@pytest.mark.parametrize("few, per", [(31, 35), (47, 50)])   # traces a bin: one part and two, two and three
@pytest.mark.parametrize("dim", [2, 3])
def test_captured_parts(vel, weight, dtype, few, per, dim):
    nb = 4
    s = sv.survey_random(np.random.default_rng(2), dim, per * nb, 70 if dim == 2 else 21, 19, 35, 200, vel=vel,
                         weight=weight, n_bins=nb, h=10.0, v0=1700.0, k=0.5 if vel == "linear" else 0.0)
    if vel == "pstm":
        s = s.replace(dz=0.01)   # two-way vertical time
    d = torch.as_tensor(sv.random_traces(s, 3, smooth=5), device="cuda").to(dtype)
    hdr, small = kh.Headers.of(s), kh.Headers.of(s.subset(np.arange(few * nb)))
    plan, other = kh.Plan(s, trace_dtype=dtype), kh.Plan(s, trace_dtype=dtype)
    plan.migrate(small, d[:few * nb].contiguous())
    got = torch.full(plan.image_shape, float("nan"), device="cuda")
    _captured(lambda: plan.migrate(hdr, d, got))
    plan.sync()
    want = other.migrate(hdr, d)
    assert torch.count_nonzero(want) > 0 and torch.equal(got, want)


@pytest.mark.parametrize("mode", ["persistent", "concurrent"])
@pytest.mark.parametrize("vel", ["const", "linear"])
def test_batch_without_room(mode, vel):
    # 40 jobs whose partial images take 0.7 GB and all else 0.3 GB, with 0.6 GB left
    def survey(ntr, n, nb, seed):
        return sv.survey_random(np.random.default_rng(seed), 3, ntr, n, n, 48, 200, vel=vel, weight="obliq", aperture=250.0,
                                n_bins=nb, h=10.0, v0=1700.0, k=0.5 if vel == "linear" else 0.0)

    kinds = []
    for i, (ntr, n, nb) in enumerate([(4000, 64, 8), (3000, 60, 8), (500, 33, 1), (40, 20, 2)]):
        s = survey(ntr, n, nb, i)
        p = kh.Plan(s)
        h, d = kh.Headers.of(s), torch.as_tensor(sv.random_traces(s, i, smooth=5), device="cuda")
        kinds.append((p, h, d, p.migrate(h, d)))
    pick = [0, 1] * 20 + [2, 3]
    jobs = [(kinds[i][0], kinds[i][1], kinds[i][2], torch.full_like(kinds[i][3], float("nan"))) for i in pick]
    roomy = kh.Batch(jobs, mode=mode)   # the kernels are loaded while there is room
    roomy.run()
    roomy.sync()
    roomy.close()
    for j in jobs:
        j[3].fill_(float("nan"))
    torch.cuda.empty_cache()
    hog = torch.empty(torch.cuda.mem_get_info()[0] - 600_000_000, dtype=torch.uint8, device="cuda")
    try:
        b = kh.Batch(jobs, mode=mode)
        used = torch.cuda.mem_get_info()[0]
        b.run()
        b.sync()
        b.run()   # the images start from the first part again
        b.sync()
    finally:
        del hog
        torch.cuda.empty_cache()
    assert used > 150_000_000   # the partial images were not held
    for i, j in zip(pick, jobs):
        assert torch.equal(j[3], kinds[i][3])
    b.close()
