"""A detector of some millions of bins: more chunks of bins than a grid's second dimension
holds.  Both projectors agree with the oracle."""
import numpy as np
import pytest

import oracle
from gpu_common import TOL, rel_l2, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "bf16", "f64"])
@pytest.mark.parametrize("N", [2, 3])
def test_projectors(N, dtype):
    from paper_1810_03275_gb300 import ctrecon as ct
    n, M = 8, 4200001
    plan = ct.Plan(n, N, M, dtype=dtype)
    rng = np.random.default_rng(N)
    u, g = rng.standard_normal((n, n)), rng.standard_normal((N, M))
    u, g = to_dev(u, plan.op_dtype), to_dev(g, plan.op_dtype)
    geo = oracle.Geometry(n, N, M)
    tol = TOL["f64" if dtype == "f64" else "f32"]
    # (FP64 at this length: coordinates in 2^-39 bins)
    tol = max(tol, 1e-9)
    assert rel_l2(to_np(plan.rh_forward(u)), oracle.rh_forward(to_np(u), geo)) < tol
    assert rel_l2(to_np(plan.rh_adjoint(g)), oracle.rh_adjoint(to_np(g), geo)) < tol
