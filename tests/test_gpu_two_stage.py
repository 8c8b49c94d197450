"""The preconditioner's two-stage transforms (FP32, n = L V with L, V <= 32): M^{-1} y against
the oracle's FFT and Alg. 4 iterations against the CTA-level passes, for every size that has one."""
import numpy as np
import pytest

import oracle
from gpu_common import rel_l2, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ct():
    from paper_1810_03275_gb300 import ctrecon
    return ctrecon


@pytest.mark.parametrize("n", [64, 72, 96, 108, 128, 144, 192, 216, 288, 324, 384, 432, 576, 648, 768, 864])
def test_two_stage_transform(ct, n):
    import torch
    sigma, tau, c, eps = 1.3, 0.35, 0.7, np.pi / n
    prm = ct.default_params(sigma=sigma, tau=tau, c=c, eps=eps)
    N, M = 8, int(np.ceil(np.sqrt(2) * n))
    plan = ct.Plan(n, N, M, angles=np.arange(N) * (np.pi / N))
    y = np.random.default_rng(n).standard_normal((n, n))
    ref = oracle.precond_apply(y, oracle.precond_symbol(n, sigma, tau, c, eps))
    assert plan.fft_form == 0
    # each of the transform's <= 14 levels of additions rounds to 2^-24: 2 x 14 x 2^-24 = 1.7e-6
    assert rel_l2(to_np(plan.precond_apply(to_dev(y, torch.float32), prm)), ref) < 2e-6
    # an input that starts in the middle of a 16-byte word takes the other passes
    z = torch.empty(n * n + 1, device="cuda")[1:].view(n, n)
    z.copy_(to_dev(y, torch.float32))
    assert rel_l2(to_np(plan.precond_apply(z, prm)), ref) < 2e-6
    # the fold of the backprojection's planes, u += ..., and Richardson's operands
    f = to_dev(np.random.default_rng(n + 1).standard_normal((N, M)), torch.float32)
    mask = (torch.rand(N, M, device="cuda", generator=torch.Generator("cuda").manual_seed(n)) < 0.05).to(torch.uint8)
    us = []
    for form in (0, 1):
        plan.set_fft_form(form)
        us.append(to_np(plan.tv_pd_solve(f, mask, 0.3, 0.05, 6,
                                         params=ct.default_params(beta=float(M), c=1.0, eps=eps))[0]))
    assert rel_l2(us[0], us[1]) < 2e-6
