"""The forward projector's launch shape: a plan reports the shape it launches, by the library's
choice or set, and every shape can be set, (1, 4) on a large plan among them."""
import pytest

from gpu_common import rel_l2, to_np

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,N,M,auto", [(64, 90, 95, (1, 4)), (512, 1440, 729, (2, 4)), (512, 1441, 729, (2, 2))])
def test_reported_and_set(n, N, M, auto):
    import torch
    from paper_1810_03275_gb300 import ctrecon as ct
    plan = ct.Plan(n, N, M)
    assert plan.symmetric_jobs > 0
    assert plan.fwd_shape == auto
    u = torch.rand((n, n), device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    chosen = plan.rh_forward(u)
    plan.set_fwd_shape(*plan.fwd_shape)
    assert torch.equal(plan.rh_forward(u), chosen)
    plan.set_fwd_shape(1, 4)
    assert plan.fwd_shape == (1, 4)
    single = plan.rh_forward(u)
    assert rel_l2(to_np(single), to_np(chosen)) < 2e-6
    # two adjacent jobs share the narrower one's chunk width, so some chunks start elsewhere
    assert torch.equal(single, chosen) == (auto == (1, 4))
