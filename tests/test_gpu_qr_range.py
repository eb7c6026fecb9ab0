"""Columns of S A V_m whose squared norms leave the range of a double in the
whitening QR: with f(z) = 1 / (1 + z) and ||A|| far below the rounding of 1,
f(A)b = b whatever the QR makes of S A V_m beside S V_m, as long as its columns
stay finite (x = V z with z from the first column alone: 1e-12)."""
import pytest
import torch

from workloads import convdiff_2d, gaussian_rhs
from workloads.operators import CSR
from gpu_helpers import rel, upload

pytestmark = pytest.mark.gpu


# norms of about 1e4 times the scale: squares normal, subnormal, and gone
@pytest.mark.parametrize("scale", [1e-140, 1e-158, 1e-160, 1e-164])
@pytest.mark.parametrize("method", ["sfom", "sgmres"])
def test_tiny_operator_in_the_full_form(skf, method, scale):
    A = convdiff_2d(40, (60.0, 50.0))
    op = upload(skf, CSR(A.n, A.rowptr, A.colind, A.values * scale))
    b = gaussian_rhs(A.n, 5)
    S = skf.Sketch(skf.SPARSE_SIGN, A.n, 96, 8, 13)
    f = skf.make_func("invsqrt", 1.0, nodes=[1.0], weights=[1.0])
    info = skf.new_info()
    with skf.tail_form(skf.TAIL_FULL), skf.arnoldi_mode(skf.ARNOLDI_TWO_KERNEL):
        x = skf.solve(skf.SFOM if method == "sfom" else skf.SGMRES, op.csr, S, torch.as_tensor(b, device="cuda"), f,
                      skf.make_params(12, 2), info=info)
    torch.cuda.synchronize()
    assert skf.read_info(info)["status"] == 0
    assert rel(x.cpu().numpy(), b) < 1e-12
