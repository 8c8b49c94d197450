"""Device memory of an FP64 plan on the symmetric path: the partial planes of its job groups (four
per group) are all that it holds beyond an angle-by-angle plan of the same sizes, with the orbit
image and the job table."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,N", [(128, 512), (256, 720), (512, 600)])
def test_no_partial_images_beside_the_partial_planes(n, N):
    from paper_1810_03275_gb300 import ctrecon as ct
    M = int(1.42 * n) + 1
    golden = np.mod(np.arange(N) * (np.pi * (np.sqrt(5.0) - 1.0) / 2.0), np.pi)
    each = 8 * n * n
    per_angle = ct.Plan(n, N, M, angles=golden, dtype="f64").device_bytes
    symmetric = ct.Plan(n, N, M, dtype="f64").device_bytes
    groups = 8                                     # both plans have room for the most
    orbit_image = 2 * 16 * n * (n + 80)
    jobs = 256 * N
    assert symmetric - per_angle <= 3 * groups * each + orbit_image + jobs
