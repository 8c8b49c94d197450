"""The FP64 symmetric projectors against the oracle where their tiling can go wrong: one pixel,
ragged images around the 16- and 32-pixel tiles, tiny and over-wide detectors, even and odd view
counts, single-view groups, bins wider than pixels; and that the pair stays adjoint."""
import numpy as np
import pytest

import oracle
from gpu_common import TOL, rel_l2, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,N,M,ds", [(1, 4, 3, 1.0), (15, 9, 23, 1.0), (17, 64, 9, 1.0), (33, 65, 300, 1.0),
                                      (64, 90, 95, 1.0), (65, 7, 93, 1.3), (130, 261, 185, 1.0), (100, 360, 60, 1.4)])
def test_matches_oracle(n, N, M, ds):
    from paper_1810_03275_gb300 import ctrecon as ct
    plan = ct.Plan(n, N, M, ds=ds, dtype="f64")
    geo = oracle.Geometry(n, N, M, ds=ds)
    rng = np.random.default_rng(n * N)
    u, g = rng.standard_normal((n, n)), rng.standard_normal((N, M))
    ru = to_np(plan.rh_forward(to_dev(u, plan.torch_dtype)))
    assert rel_l2(ru, oracle.rh_forward(u, geo)) < TOL["f64"]
    for groups in sorted({1, plan.bp_groups}):
        plan.set_bp_groups(groups)
        rtg = to_np(plan.rh_adjoint(to_dev(g, plan.torch_dtype)))
        assert rel_l2(rtg, oracle.rh_adjoint(g, geo)) < TOL["f64"]
    # 1e-13: rounding of the two inner products, some 1e5 terms
    assert abs(np.vdot(ru, g) - np.vdot(u, rtg)) < 1e-13 * np.linalg.norm(ru) * np.linalg.norm(g) + 1e-300
