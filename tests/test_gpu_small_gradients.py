"""The adjoint's traveltimes at small velocity gradients, where ln(u) of a leg is far below 1 and is divided
by |k| dt: against the oracle, and as the transpose of the migration."""
import numpy as np
import pytest

import oracle
from helpers import FP32_REL_L2, gpu_demigrate, gpu_migrate, rel_l2
from paper_1204_1225_gb300 import survey as sv

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1e-1, 1e-2, -1e-2, 1e-3, 1e-4, -1e-5, 1e-6, 1e-7, -1e-8, 1e-8])
@pytest.mark.parametrize("dim", [2, 3])
def test_small_gradients(k, dim):
    rng = np.random.default_rng(31)
    s = sv.survey_random(rng, dim, 130, 22, 18, 40, 402, vel="linear", weight="obliq", n_bins=2, h=12.5, v0=1800.0, k=k)
    d = sv.random_traces(s, 1, smooth=5)
    # a migrated image: a white-noise one makes samples of random-sign terms, whose rounding is near the bar
    m = oracle.migrate(s, d).astype(np.float32)
    got, p = gpu_demigrate(s, m)
    assert rel_l2(got, oracle.demigrate(s, m)) < FP32_REL_L2
    Ld, _ = gpu_migrate(s, d, plan=p)
    lhs, rhs = float(np.vdot(Ld, m.astype(np.float64))), float(np.vdot(d.astype(np.float64), got))
    assert abs(lhs - rhs) <= 1e-5 * max(abs(lhs), abs(rhs))
