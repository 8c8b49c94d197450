"""The block form of the symmetric backprojection against the oracle where its tiling can go
wrong: one pixel, ragged tiles, image widths that are and are not multiples of 2 and 4, tiny
and over-wide detectors, even view counts (four-channel jobs) and odd ones (pair jobs), job
counts around the table and chunk sizes, and bins wider than pixels."""
import numpy as np
import pytest

import oracle
from gpu_common import TOL, rel_l2, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ct():
    from paper_1810_03275_gb300 import ctrecon
    return ctrecon


@pytest.mark.parametrize("n,N,M,ds", [(1, 4, 3, 1.0), (2, 4, 1, 1.0), (31, 63, 45, 1.0), (33, 65, 9, 1.0),
                                      (34, 128, 49, 1.0), (66, 130, 400, 1.3), (97, 1030, 138, 1.0),
                                      (64, 261, 91, 1.4), (36, 1029, 52, 1.0)])
@pytest.mark.parametrize("dtype", ["f32", "bf16"])
def test_matches_oracle(ct, n, N, M, ds, dtype):
    import torch
    plan = ct.Plan(n, N, M, ds=ds, dtype=dtype)
    assert plan.symmetric_jobs > 0
    g = to_dev(np.random.default_rng(n * N).standard_normal((N, M)), plan.op_dtype)
    want = oracle.rh_adjoint(to_np(g), oracle.Geometry(n, N, M, ds=ds))
    for groups in sorted({1, plan.bp_groups}):
        plan.set_bp_groups(groups)
        assert rel_l2(to_np(plan.rh_adjoint(g)), want) < TOL["f32"]
    torch.cuda.synchronize()
