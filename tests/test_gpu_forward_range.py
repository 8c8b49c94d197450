"""The forward projector over the whole FP32 range: images whose projections are representable
project finitely, whatever their scale (no intermediate is larger than the sum of the pixels)."""
import numpy as np
import pytest

import oracle
from gpu_common import TOL, rel_l2, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [60, 61])
@pytest.mark.parametrize("scale", [1e-25, 1e30, 1e35])
def test_scales_with_the_image(N, scale):
    import torch
    from paper_1810_03275_gb300 import ctrecon as ct
    n, M = 65, 95
    plan = ct.Plan(n, N, M)
    assert plan.symmetric_jobs > 0
    u = np.random.default_rng(N).uniform(0.0, 1.0, (n, n)).astype(np.float32)
    got = to_np(plan.rh_forward(to_dev(u * np.float32(scale), torch.float32)))
    want = oracle.rh_forward((u * np.float32(scale)).astype(np.float64), oracle.Geometry(n, N, M))
    assert np.isfinite(got).all()
    assert rel_l2(got / scale, want / scale) < TOL["f32"]
