"""Each view of the ramp filter comes out as it would alone, whatever stands beside it: views of
comparable maxima and very different energies (a wide view beside a narrow pin), to a rounding
that its own norm bounds, and bit for bit independent of the neighbour."""
import numpy as np
import pytest

import oracle
from gpu_common import to_dev, to_np

pytestmark = pytest.mark.gpu

# Two transforms of at most 2^12 points, each within log2(L) roundings of its input's norm, and a
# multiplier of at most 1/2 between them: 2 x 12 x 2^-24 / 2 (2^-53 in FP64) of the view's norm
BOUND = {"f32": 1e-6, "f64": 2e-15}


def _views(M):
    s = np.arange(M) - 0.5 * (M - 1)
    disk = 2.0 * np.sqrt(np.maximum((0.4 * M) ** 2 - s ** 2, 0.0))
    pin, spike, flat = np.zeros(M), np.zeros(M), np.ones(M)
    pin[M // 3:M // 3 + 5] = 1.0
    spike[M // 2] = 1.0
    rough = np.random.default_rng(M).standard_normal(M)
    return {"disk": disk / disk.max(), "pin": pin, "spike": spike, "flat": flat, "rough": rough}


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("M", [95, 729, 1449])
@pytest.mark.parametrize("ratio", [1.0, 8.0, 60.0])
def test_accuracy_of_each_view(M, ratio, dtype):
    from paper_1810_03275_gb300 import ctrecon as ct
    v = _views(M)
    big, small = ("disk", "flat", "rough"), ("pin", "spike", "rough")
    g = np.stack([x for b in big for s in small for x in (ratio * v[b], v[s])])
    plan = ct.Plan(16, len(g), M, dtype=dtype)
    dev = to_dev(g, plan.torch_dtype)
    y, ref = to_np(plan.ramp_filter(dev)), oracle.ramp_filter(to_np(dev))
    for l in range(len(g)):
        assert np.linalg.norm(y[l] - ref[l]) < BOUND[dtype] * np.linalg.norm(g[l]), l


@pytest.mark.parametrize("M", [1, 2, 60, 95, 730, 1449])
def test_independent_of_the_neighbour(M):
    import torch
    from paper_1810_03275_gb300 import ctrecon as ct
    plan = ct.Plan(16, 3, M)
    rng = np.random.default_rng(M)
    g = to_dev(rng.standard_normal((3, M)), torch.float32)
    first = plan.ramp_filter(g).clone()
    g[1] = to_dev(5.0 * rng.standard_normal(M), torch.float32)
    second = plan.ramp_filter(g)
    assert torch.equal(first[0], second[0]) and torch.equal(first[2], second[2])
