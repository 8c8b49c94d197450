"""The transforms of a batch are shared out over thread blocks by the number of its slices: every
split gives the slices' own results (one slice, a few, and more than the blocks aimed at), for
sizes with one and with several transforms per block, even and odd half spectra."""
import numpy as np
import pytest

from gpu_common import rel_l2, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [24, 54, 64, 96, 128])
@pytest.mark.parametrize("count", [1, 3, 20, 130])
def test_slices_as_alone(n, count):
    import torch
    from paper_1810_03275_gb300 import ctrecon as ct
    N, M = 40, int(1.42 * n) + 2
    rng = np.random.default_rng(n)
    scans = [to_dev(rng.uniform(0, n, (N, M)), torch.float32) for _ in range(min(count, 3))]
    fs = [scans[i % len(scans)] for i in range(count)]
    beta, c, iters = float(np.sqrt(n * N)), 12.0 / n, 12
    batch = ct.Batch([{"n": n, "n_angles": N, "n_bins": M}] * count)
    us, _ = batch.solve(fs, None, [0.1] * count, [0.5] * count, iters, params=ct.default_params(), betas=[beta] * count,
                        cs=[c] * count, want_diag=False)
    plan = ct.Plan(n, N, M)
    for i, f in enumerate(scans):
        alone, _ = plan.tv_pd_solve(f, None, 0.1, 0.5, iters, params=ct.default_params(beta=beta, c=c))
        # (the same arithmetic in instances of their own, and other transforms where a plan has them)
        assert rel_l2(to_np(us[i]), to_np(alone)) < 2e-6
    for i in range(len(scans), count):
        assert torch.equal(us[i], us[i % len(scans)])
