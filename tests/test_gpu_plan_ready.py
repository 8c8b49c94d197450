"""A plan is ready when its creation returns: its tables and the zeros around its padded operands
are there for calls on any stream, also while the default stream, which they were written on, has
other work queued ahead of them, and in memory that held other values before."""
import numpy as np
import pytest

import oracle
from gpu_common import TOL, rel_l2, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", ["f32", "bf16", "f64"])
@pytest.mark.parametrize("N", [60, 61])
def test_first_calls_on_another_stream(N, dtype):
    import torch
    from paper_1810_03275_gb300 import ctrecon as ct
    n, M = 130, 185
    rng = np.random.default_rng(N)
    op = {"f32": torch.float32, "bf16": torch.bfloat16, "f64": torch.float64}[dtype]
    u, g = to_dev(rng.standard_normal((n, n)), op), to_dev(rng.standard_normal((N, M)), op)
    geo = oracle.Geometry(n, N, M)
    want_g, want_u = oracle.rh_forward(to_np(u), geo), oracle.rh_adjoint(to_np(g), geo)
    a = torch.randn((4096, 4096), device="cuda")
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(20):
        a = torch.tanh(a @ a)                     # some milliseconds on the default stream
    plan = ct.Plan(n, N, M, dtype=dtype)
    with torch.cuda.stream(side):
        got_g, got_u = plan.rh_forward(u), plan.rh_adjoint(g)
    side.synchronize()
    tol = TOL["f64" if dtype == "f64" else "f32"]
    assert rel_l2(to_np(got_g), want_g) < tol and rel_l2(to_np(got_u), want_u) < tol
    torch.cuda.synchronize()
