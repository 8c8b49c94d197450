"""The slot form of the symmetric forward projector against the oracle where its tiling can go
wrong: one pixel, ragged images and detectors, widths that are not a multiple of a 16-byte
unit, even view counts (four-channel jobs) and odd ones (pair jobs), views too sparse to share
staged rows and dense ones, bins wider than pixels, and every launch shape."""
import numpy as np
import pytest

import oracle
from gpu_common import TOL, rel_l2, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ct():
    from paper_1810_03275_gb300 import ctrecon
    return ctrecon


@pytest.mark.parametrize("n,N,M,ds", [(1, 4, 3, 1.0), (31, 63, 45, 1.0), (33, 64, 9, 1.0), (65, 7, 93, 1.0),
                                      (64, 8, 200, 1.0), (97, 400, 138, 1.0), (130, 261, 60, 1.4), (200, 12, 283, 1.3)])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_matches_oracle(ct, n, N, M, ds, dtype):
    plan = ct.Plan(n, N, M, ds=ds, dtype=dtype)
    assert plan.symmetric_jobs > 0
    u = to_dev(np.random.default_rng(n * N).standard_normal((n, n)), plan.op_dtype)
    want = oracle.rh_forward(to_np(u), oracle.Geometry(n, N, M, ds=ds))
    for shape in plan.FWD_SHAPES:
        plan.set_fwd_shape(*shape)
        assert rel_l2(to_np(plan.rh_forward(u)), want) < TOL["f32"], shape
