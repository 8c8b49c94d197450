"""The FP64 preconditioner on either side of the size where its transforms go from radix 2 to mixed
radices: against the same filter from 64-bit transforms."""
import numpy as np
import pytest

from gpu_common import rel_l2, to_dev, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 6, 8, 162, 216, 243, 256, 288, 512, 1024])
def test_against_64_bit_transforms(n):
    from paper_1810_03275_gb300 import ctrecon as ct
    plan = ct.Plan(n, 4, n + 1, dtype="f64")
    c, tau, eps = 12.0 / n, 1.0 / np.sqrt(8.0), np.pi / n
    y = np.random.default_rng(n).standard_normal((n, n))
    got = to_np(plan.precond_apply(to_dev(y, plan.torch_dtype), ct.default_params(c=c)))
    xi = 2 * np.pi * np.fft.fftfreq(n)
    norm = np.sqrt(xi[:, None] ** 2 + xi[None, :] ** 2 + eps ** 2)
    s = 4 * np.sin(np.pi * np.arange(n) / n) ** 2
    want = np.fft.ifft2(np.fft.fft2(y) * norm / (c + tau ** 2 * (s[:, None] + s[None, :]) * norm)).real
    # some 20 passes' roundings of 2^-53 each way: 1e-14 leaves a factor of two
    assert rel_l2(got, want) < 1e-14
