"""The metal trace holds only bins that a mark touches, down to proj_tol = 0: R_h of the 0/1
image of marks is exactly 0 elsewhere.  Long marks (their slots sum hundreds of pixels) and
small disks, symmetric plans with four-channel and with pair jobs, FP32, BF16 and FP64."""
import numpy as np
import pytest

import oracle
from gpu_common import to_dev, to_np

pytestmark = pytest.mark.gpu


def _touched(marks, theta, M):
    """Bins k with |p - k| < 1 for some marked pixel's coordinate p (1e-6 bins of slack for the
    quantised geometry)."""
    n = marks.shape[0]
    i, j = np.nonzero(marks)
    x, y = i - 0.5 * (n - 1), j - 0.5 * (n - 1)
    out = np.zeros((len(theta), M), dtype=bool)
    for l, t in enumerate(theta):
        p = x * np.cos(t) + y * np.sin(t) + 0.5 * (M - 1)
        for k in (np.floor(p - 1e-6), np.floor(p + 1e-6) + 1):
            k = k.astype(int)
            out[l, k[(k >= 0) & (k < M)]] = True
    return out


@pytest.mark.parametrize("n,N,M,dtype", [(512, 720, 729, "f32"), (512, 721, 729, "f32"), (512, 720, 729, "bf16"),
                                         (256, 360, 363, "f32"), (256, 360, 363, "f64"), (256, 361, 363, "f64")])
def test_untouched_bins_are_exactly_zero(n, N, M, dtype):
    from paper_1810_03275_gb300 import ctrecon as ct
    plan = ct.Plan(n, N, M, dtype=dtype)
    assert plan.symmetric_jobs > 0 or dtype == "f64"      # (counts FP32 and BF16 jobs)
    theta = np.arange(N) * (np.pi / N)
    u = np.zeros((n, n))
    u[n // 3:n // 3 + n // 4, n // 2:n // 2 + n // 26] = 3.0       # a long bar
    i, j = np.ogrid[:n, :n]
    u[(i - 0.7 * n) ** 2 + (j - 0.3 * n) ** 2 < 30] = 3.0          # and a small disk
    touched = _touched(u > 2, theta, M)
    dev = to_dev(u, plan.torch_dtype)
    for tol in (0.0, 1e-6):
        trace, marks = plan.metal_trace(dev, 2.0, 0, tol, want_marks=True)
        np.testing.assert_array_equal(to_np(marks) > 0, u > 2)
        assert not (to_np(trace).astype(bool) & ~touched).any()
    # and it holds every bin that the marks fill to more than the projector's rounding
    filled = oracle.rh_forward((u > 2).astype(np.float64), oracle.Geometry(n, N, M)) > 1e-3
    assert to_np(trace).astype(bool)[filled].all()
