"""Edges of the Arnoldi step kernels, the embeddings and the QR at the sizes
where their partitions, layouts and scales change: few rows per CTA, compact
and general sketch patterns, extreme magnitudes (the grid sums are exact
integers below an exponent bound), happy breakdown with every embedding in the
two-kernel form, the pruned and the full DCT, bin copies of the sketch apply.
Against the FP64 oracle, with the tolerances of the same quantities elsewhere:
1e-11 per Arnoldi column, 1e-14 for an exact sparse-sign sum, 1e-13 sqrt(N) of
the column's norm for a DCT."""
import numpy as np
import pytest
import torch

from oracle.arnoldi import arnoldi_trunc as o_arnoldi
from oracle.sketch import Sketch as OSketch
from workloads import convdiff_2d, csr_to_scipy, gaussian_rhs
from workloads.operators import CSR
from gpu_helpers import rel, upload

pytestmark = pytest.mark.gpu

KIND = {"sparse_sign": 0, "srht": 1, "srdct": 3}


def check_columns(skf, A, b, m, k, s, mode, kind="sparse_sign", zeta=8, tol=1e-11):
    op = upload(skf, A)
    S = skf.Sketch(KIND[kind], A.n, s, zeta, 13)
    info = skf.new_info()
    with skf.arnoldi_mode(mode):
        V, vs, SV, SAV, H = skf.arnoldi_trunc(op.csr, S, torch.as_tensor(b, device="cuda"), m, k, info=info)
    torch.cuda.synchronize()
    ar = o_arnoldi(csr_to_scipy(A), b, m, k, OSketch(kind, A.n, s, zeta, 13))
    info = skf.read_info(info)
    assert info["m_eff"] == ar["m_eff"]
    Vn = (V * vs[:, None]).cpu().numpy()
    for j in range(ar["m_eff"]):
        assert rel(Vn[j], ar["V"][:, j]) < tol, j
        assert rel(SV[j].cpu().numpy(), ar["SV"][:, j]) < tol, j
        assert rel(SAV[j].cpu().numpy(), ar["SAV"][:, j]) < tol, j
    nh = ar["m_eff"] - 1
    Hg, Ho = H.cpu().numpy().T[:, :nh], ar["H"][:, :nh]
    assert np.abs(Hg[: Ho.shape[0]] - Ho).max() <= tol * np.abs(Ho).max()


# one CTA, one row over, several CTAs with a ragged last one, the last size of
# 256 rows per CTA on 152 SMs and the first beyond it (38809 = 197^2 and 198^2)
@pytest.mark.parametrize("n", [3, 16, 17, 71, 197, 198])
@pytest.mark.parametrize("k", [1, 2, 4])
def test_persistent_partition_edges(skf, n, k):
    A = convdiff_2d(n, (60.0, 50.0))
    m = min(10, A.n // 2)
    check_columns(skf, A, gaussian_rhs(A.n, 3), m, k, min(4 * m, A.n), skf.ARNOLDI_PERSISTENT, zeta=min(8, m + 1))


# stripes of 64 / 65 / 128 / 129 rows (compact pattern with one byte and either
# sign offset, general pattern), and a sparsity without the compact pattern
@pytest.mark.parametrize("s,zeta", [(512, 8), (520, 8), (1024, 8), (1032, 8), (300, 5), (200, 16)])
@pytest.mark.parametrize("form", ["persistent", "two_kernel"])
def test_bin_layouts(skf, s, zeta, form):
    A = convdiff_2d(61, (60.0, 50.0))
    mode = skf.ARNOLDI_PERSISTENT if form == "persistent" else skf.ARNOLDI_TWO_KERNEL
    check_columns(skf, A, gaussian_rhs(A.n, 4), 9, 2, s, mode, zeta=zeta)


@pytest.mark.parametrize("sa,sb", [(1e60, 1.0), (1e-60, 1.0), (1.0, 1e120), (1.0, 1e-120), (1e40, 1e-80)])
@pytest.mark.parametrize("form", ["persistent", "two_kernel"])
def test_magnitudes(skf, sa, sb, form):
    A = convdiff_2d(70, (60.0, 50.0))
    A = CSR(A.n, A.rowptr, A.colind, A.values * sa)
    mode = skf.ARNOLDI_PERSISTENT if form == "persistent" else skf.ARNOLDI_TWO_KERNEL
    check_columns(skf, A, gaussian_rhs(A.n, 5) * sb, 12, 2, 64, mode)


def test_dots_of_a_near_null_vector(skf):
    """||A||_inf is set by one row that b avoids, so the bound of the dot
    products lies 1e12 above their values."""
    n = 60
    A = convdiff_2d(n, (60.0, 50.0))
    vals = A.values.copy()
    last = slice(int(A.rowptr[A.n - 1]), int(A.rowptr[A.n]))
    vals[last] *= 1e12
    b = gaussian_rhs(A.n, 6)
    b[-2 * n - 2:] = 0.0
    check_columns(skf, CSR(A.n, A.rowptr, A.colind, vals), b, 2, 2, 32, skf.ARNOLDI_PERSISTENT)


@pytest.mark.parametrize("form", ["persistent", "two_kernel"])
def test_non_finite_operator_entry_ends_the_process(skf, form):
    """An infinite product makes the dot products NaN: no vector follows."""
    A = convdiff_2d(50, (60.0, 50.0))
    vals = A.values.copy()
    vals[777] = np.inf
    op = upload(skf, CSR(A.n, A.rowptr, A.colind, vals))
    S = skf.Sketch(skf.SPARSE_SIGN, A.n, 40, 8, 13)
    info = skf.new_info()
    with skf.arnoldi_mode(skf.ARNOLDI_PERSISTENT if form == "persistent" else skf.ARNOLDI_TWO_KERNEL):
        skf.arnoldi_trunc(op.csr, S, torch.as_tensor(gaussian_rhs(A.n, 1), device="cuda"), 8, 2, info=info)
    torch.cuda.synchronize()
    info = skf.read_info(info)
    assert info["m_eff"] == 1 and info["breakdown"] == 1


# the noise vector w_{m_eff} closes the last relation: S A v_{m_eff - 1} is as
# accurate as the others with every embedding
@pytest.mark.parametrize("kind", ["sparse_sign", "srht", "srdct"])
@pytest.mark.parametrize("m", [5, 6, 12])
def test_two_kernel_happy_breakdown(skf, kind, m):
    lam = np.repeat([1.0, 2.0, 3.5, 7.0, 11.0], 300)
    N = lam.size
    A = CSR(N, np.arange(N + 1, dtype=np.int64), np.arange(N, dtype=np.int32), lam)
    check_columns(skf, A, gaussian_rhs(N, 5), m, 2, 60, skf.ARNOLDI_TWO_KERNEL, kind=kind,
                  zeta=8 if kind == "sparse_sign" else 0)


# L = N / 2 = 512 (one group), 4608 = 512 x 9 and 62500 = 1000-limit groups with
# few samples (pruned) and all (full passes), odd N
@pytest.mark.parametrize("N,s", [(1024, 64), (9216, 100), (9216, 9216), (125000, 200), (4725, 50), (3 ** 9, 400)])
def test_srdct_pruned_and_full(skf, N, s):
    X = np.random.default_rng(N + s).standard_normal((N, 3))
    S = skf.Sketch(skf.SRDCT, N, s, 0, 17)
    SX = skf.sketch_apply(S, torch.as_tensor(X, device="cuda")).cpu().numpy()
    SO = OSketch("srdct", N, s, seed=17) @ X
    for c in range(3):
        assert np.linalg.norm(SX[:, c] - SO[:, c]) <= 1e-13 * np.sqrt(N) * np.linalg.norm(X[:, c])


# 16 bin copies up to s = 864, fewer beyond, one for the largest; compact and
# general pattern; a zero column and a column with one entry
@pytest.mark.parametrize("N,s,zeta", [(31, 8, 8), (4096, 864, 8), (4096, 872, 8), (20_011, 1600, 8),
                                      (20_011, 1600, 5), (30_000, 12_000, 8)])
def test_sketch_apply_bin_copies(skf, N, s, zeta):
    X = np.random.default_rng(N).standard_normal((N, 5))
    X[:, 1] = 0.0
    X[:, 3] = 0.0
    X[N - 1, 3] = -1e-7
    S = skf.Sketch(skf.SPARSE_SIGN, N, s, zeta, 21)
    got = skf.sketch_apply(S, torch.as_tensor(X, device="cuda")).cpu().numpy()
    want = OSketch("sparse_sign", N, s, zeta, 21) @ X
    assert not got[:, 1].any()
    for c in (0, 2, 3, 4):
        assert np.linalg.norm(got[:, c] - want[:, c]) <= 1e-14 * np.linalg.norm(want[:, c])
