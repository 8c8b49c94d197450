"""NaN and infinite operands of the projectors stay where the interpolation puts them: a pixel
reaches the two bins around its coordinate in each view, a bin the pixels whose coordinate lies
within one bin of it, and everything else comes out as if the value were absent."""
import numpy as np
import pytest

import oracle
from gpu_common import to_dev, to_np

pytestmark = pytest.mark.gpu

GEOMS = [(64, 90, 95, 1.0), (48, 61, 71, 1.3), (300, 64, 427, 1.0), (270, 45, 400, 1.0)]
BOUND = {"f32": 1e-5, "bf16": 1e-5, "f64": 1e-10}
SLACK = 1e-6           # bins: the fixed-point geometry's quantisation


def _coords(n, theta, M, ds):
    x = np.arange(n) - 0.5 * (n - 1)
    c, s = np.cos(theta)[:, None, None], np.sin(theta)[:, None, None]
    return (x[:, None] * c + x[None, :] * s) / ds + 0.5 * (M - 1)


def _check(got, want, must, may, bound):
    bad = ~np.isfinite(got)
    assert not (bad & ~may).any() and bad[must].all()
    ok = ~bad
    assert np.abs(got - want)[ok].max() < bound * np.abs(want).max()


@pytest.mark.parametrize("dtype", ["f32", "bf16", "f64"])
@pytest.mark.parametrize("n,N,M,ds", GEOMS)
@pytest.mark.parametrize("value", [np.nan, -np.inf])
def test_forward(n, N, M, ds, dtype, value):
    from paper_1810_03275_gb300 import ctrecon as ct
    plan = ct.Plan(n, N, M, ds=ds, dtype=dtype)
    assert plan.symmetric_jobs > 0 or dtype == "f64"      # (counts FP32 and BF16 jobs)
    theta = np.arange(N) * (np.pi / N)
    u = np.random.default_rng(n).standard_normal((n, n))
    i, j = n // 3, (2 * n) // 5
    u = to_np(to_dev(u, plan.op_dtype))
    u[i, j] = 0.0
    want = oracle.rh_forward(u, oracle.Geometry(n, N, M, ds=ds))
    u[i, j] = value
    got = to_np(plan.rh_forward(to_dev(u, plan.op_dtype)))
    p = _coords(n, theta, M, ds)[:, i, j][:, None]
    k = np.arange(M)[None, :]
    must = (k == np.floor(p + SLACK)) & (k == np.floor(p - SLACK))
    may = (k >= np.floor(p - SLACK)) & (k <= np.floor(p + SLACK) + 1)
    _check(got, want, must, may, BOUND[dtype])


@pytest.mark.parametrize("dtype", ["f32", "bf16", "f64"])
@pytest.mark.parametrize("n,N,M,ds", GEOMS)
@pytest.mark.parametrize("value", [np.nan, np.inf])
def test_adjoint(n, N, M, ds, dtype, value):
    from paper_1810_03275_gb300 import ctrecon as ct
    plan = ct.Plan(n, N, M, ds=ds, dtype=dtype)
    assert plan.symmetric_jobs > 0 or dtype == "f64"      # (counts FP32 and BF16 jobs)
    theta = np.arange(N) * (np.pi / N)
    g = to_np(to_dev(np.random.default_rng(n).standard_normal((N, M)), plan.op_dtype))
    spots = [(0, M // 2), (N // 6, M // 2 + 7), (N - 3, M // 2 - 9)]      # flat and steep views
    for l, k in spots:
        g[l, k] = 0.0
    want = oracle.rh_adjoint(g, oracle.Geometry(n, N, M, ds=ds))
    must = np.zeros((n, n), dtype=bool)
    may = must.copy()
    p = _coords(n, theta, M, ds)
    for l, k in spots:
        g[l, k] = value
        must |= np.abs(p[l] - k) < 1 - SLACK
        may |= np.abs(p[l] - k) < 1 + SLACK
    got = to_np(plan.rh_adjoint(to_dev(g, plan.op_dtype)))
    _check(got, want, must, may, BOUND[dtype])
