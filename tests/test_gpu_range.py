"""Operators whose scale takes the products of a step out of the range of a
double: the process ends with the columns it has, and those columns are right."""
import numpy as np
import pytest
import torch

from oracle.sketch import Sketch as OSketch
from workloads import convdiff_2d, csr_to_scipy, gaussian_rhs
from workloads.operators import CSR
from gpu_helpers import rel, upload

pytestmark = pytest.mark.gpu

KIND = {"sparse_sign": 0, "srht": 1, "srdct": 3}


def columns(skf, form, scale, kind="sparse_sign", m=6):
    A = convdiff_2d(40, (60.0, 50.0))
    A = CSR(A.n, A.rowptr, A.colind, A.values * scale)
    op = upload(skf, A)
    zeta = 8 if kind == "sparse_sign" else 0
    S = skf.Sketch(KIND[kind], A.n, 96, zeta, 13)
    info = skf.new_info()
    with skf.arnoldi_mode(skf.ARNOLDI_PERSISTENT if form == "persistent" else skf.ARNOLDI_TWO_KERNEL):
        V, vs, SV, SAV, H = skf.arnoldi_trunc(op.csr, S, torch.as_tensor(gaussian_rhs(A.n, 5), device="cuda"), m, 2,
                                              info=info)
    torch.cuda.synchronize()
    return A, OSketch(kind, A.n, 96, zeta, 13), (V * vs[:, None]).cpu().numpy(), SAV.cpu().numpy(), skf.read_info(info)


# ||A v|| about 1e134 and 1e149: the dot products of the second step overflow, so
# w_2 is not a number and the process ends with two columns
@pytest.mark.parametrize("scale", [1e130, 1e145])
@pytest.mark.parametrize("form,kind", [("persistent", "sparse_sign"), ("two_kernel", "sparse_sign"),
                                       ("two_kernel", "srht"), ("two_kernel", "srdct")])
def test_last_column_of_an_overflowing_process(skf, form, kind, scale):
    A, S, V, SAV, info = columns(skf, form, scale, kind)
    assert info["breakdown"] == 1 and info["m_eff"] == 2
    for j in range(2):
        assert rel(SAV[j], S @ (csr_to_scipy(A) @ V[j])) < 1e-11, j


# the default tail on it: x = A^{-1}-like values, finite, status OK
@pytest.mark.parametrize("form", ["persistent", "two_kernel"])
def test_solve_of_an_overflowing_process(skf, form):
    A = convdiff_2d(40, (60.0, 50.0))
    op = upload(skf, CSR(A.n, A.rowptr, A.colind, A.values * 1e130))
    S = skf.Sketch(skf.SPARSE_SIGN, A.n, 96, 8, 13)
    b = torch.as_tensor(gaussian_rhs(A.n, 5), device="cuda")
    f = skf.make_func("invsqrt", 1.0, nodes=[1e134], weights=[1.0])
    for method in (skf.SFOM, skf.SGMRES):
        info = skf.new_info()
        with skf.arnoldi_mode(skf.ARNOLDI_PERSISTENT if form == "persistent" else skf.ARNOLDI_TWO_KERNEL):
            x = skf.solve(method, op.csr, S, b, f, skf.make_params(6, 2), info=info)
        torch.cuda.synchronize()
        assert skf.read_info(info)["status"] == 0
        assert 0.0 < float(x.norm()) * 1e134 < float(b.norm())


# ||w_1||^2 about 1e-308 and below: its summands are subnormal; the second step's
# norm is gone and ends the process in both forms
@pytest.mark.parametrize("form", ["persistent", "two_kernel"])
@pytest.mark.parametrize("scale", [1e-158, 1e-160])
def test_subnormal_norms_count(skf, form, scale):
    A, S, V, SAV, info = columns(skf, form, scale)
    assert info["breakdown"] == 1 and info["m_eff"] == 2
    assert rel(SAV[0], S @ (csr_to_scipy(A) @ V[0])) < 1e-11
