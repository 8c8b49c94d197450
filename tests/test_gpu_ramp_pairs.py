"""The ramp filter transforms two views as one complex sequence: odd view counts, views of very
different size, blank views and views with non-finite values must come out as each view alone
would, and detectors around the lengths where the transform length changes match the oracle."""
import numpy as np
import pytest

import oracle
from gpu_common import TOL, rel_l2, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("N,M", [(1, 1), (2, 2), (3, 61), (5, 513), (4, 730), (7, 1449)])
def test_matches_oracle(N, M, dtype):
    from paper_1810_03275_gb300 import ctrecon as ct
    plan = ct.Plan(16, N, M, dtype=dtype)
    g = np.random.default_rng(M).standard_normal((N, M))
    y = to_np(plan.ramp_filter(to_dev(g, plan.torch_dtype)))
    assert rel_l2(y, oracle.ramp_filter(g)) < TOL[dtype]


def test_views_do_not_touch_each_other():
    import torch
    from paper_1810_03275_gb300 import ctrecon as ct
    N, M = 6, 95
    plan = ct.Plan(16, N, M)
    g = np.random.default_rng(2).standard_normal((N, M))
    g[1] = 0.0                       # beside an ordinary view
    g[2] *= 1e6                      # beside one a million times smaller
    g[4, 7], g[4, 50] = np.inf, np.nan
    y = to_np(plan.ramp_filter(to_dev(g, torch.float32)))
    ref = oracle.ramp_filter(np.nan_to_num(g, nan=0.0, posinf=0.0))
    assert np.all(y[1] == 0.0)
    for v in (0, 2, 3, 5):
        assert rel_l2(y[v], ref[v]) < TOL["f32"], v
    assert not np.isfinite(y[4]).any()
