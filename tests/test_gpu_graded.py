"""Operators whose ||A||_inf lies far above the products: one decoupled row
carries the norm and the right-hand side vanishes there, so every A v_j is that
of the other rows.  The persistent form sums its dot products as integers below
an exponent bound that holds ||A||_inf; the columns still have to agree with the
FP64 oracle (1e-11 per column, as elsewhere), and those of an FP32 basis with
the same operator without the large row (1e-5: m = 8 steps of FP32 rounding)."""
import numpy as np
import pytest
import torch

from workloads import convdiff_2d, gaussian_rhs
from workloads.operators import CSR
from gpu_helpers import rel
from test_gpu_step_edges import check_columns

pytestmark = pytest.mark.gpu


def with_decoupled_row(n, big):
    A = convdiff_2d(n, (60.0, 50.0))
    return CSR(A.n + 1, np.append(A.rowptr, A.rowptr[-1] + 1), np.append(A.colind, np.int32(A.n)),
               np.append(A.values, big))


def rhs(N):
    return np.append(gaussian_rhs(N - 1, 5), 0.0)


# 1e18: the bound as it is (60 bits above the products), 1e30 and 1e45: beyond
# what the sums keep below it
@pytest.mark.parametrize("big", [1e18, 1e30, 1e45])
@pytest.mark.parametrize("n,k", [(40, 1), (40, 2), (40, 4), (200, 2)])
def test_decoupled_row_carries_the_norm(skf, n, k, big):
    A = with_decoupled_row(n, big)
    check_columns(skf, A, rhs(A.n), 12, k, 64, skf.ARNOLDI_PERSISTENT)


@pytest.mark.parametrize("form", ["persistent", "two_kernel"])
def test_decoupled_row_fp32_basis(skf, form):
    m, out = 8, []
    for big in (1.0, 1e38):
        A = with_decoupled_row(60, big)
        op = skf.upload_csr(A.rowptr, A.colind, A.values.astype(np.float32), device="cuda")
        S = skf.Sketch(skf.SPARSE_SIGN, A.n, 64, 8, 13)
        with skf.arnoldi_mode(skf.ARNOLDI_PERSISTENT if form == "persistent" else skf.ARNOLDI_TWO_KERNEL):
            V, vs, *_ = skf.arnoldi_trunc(op.csr, S, torch.as_tensor(rhs(A.n), device="cuda"), m, 2,
                                          basis_dtype=torch.float32)
        torch.cuda.synchronize()
        out.append((V.double() * vs[:, None]).cpu().numpy())
    for j in range(m):
        assert rel(out[1][j], out[0][j]) < 1e-5, j
