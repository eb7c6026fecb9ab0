"""The last Arnoldi step with an SRDCT transforms w_j and A w_j in one set of
launches: with full FFT passes (many samples) a step is bound by its launches."""
import pytest
import torch

from workloads import convdiff_2d, gaussian_rhs
from gpu_helpers import upload

pytestmark = pytest.mark.gpu


def test_last_step_takes_no_second_set_of_launches(skf):
    A = convdiff_2d(200, (60.0, 50.0))
    op = upload(skf, A)
    S = skf.Sketch(skf.SRDCT, A.n, 1200, 0, 13)
    b = torch.as_tensor(gaussian_rhs(A.n, 3), device="cuda")

    def launches(m):
        n0 = skf.kernel_launch_count()
        skf.arnoldi_trunc(op.csr, S, b, m, 2)
        return skf.kernel_launch_count() - n0

    step = (launches(4) - launches(2)) // 2
    assert step >= 10   # the product, the update, the reordering, the passes, the gather
    assert launches(2) - 2 * step <= 6   # start, finish, estimate, info
