"""Small solves beside each other (skf_solve_batched): on many lanes they take
fewer CTAs each, and two CTAs fit on an SM.  Whatever the partition, a problem
gives the bits of its own skf_solve call, for every form of the persistent
kernel (basis type, window, row width, pattern), and the lanes overlap."""
import numpy as np
import pytest
import torch

from oracle.arnoldi import arnoldi_trunc as o_arnoldi
from oracle.sketch import Sketch as OSketch
from workloads import convdiff_2d, convdiff_3d, csr_to_scipy, gaussian_rhs
from workloads.operators import CSR
from gpu_helpers import rel, upload

pytestmark = pytest.mark.gpu


def wide(n, width, seed):
    """n rows of `width` entries on random circulant diagonals, diagonally dominant."""
    g = np.random.default_rng(seed)
    off = np.append(0, 1 + g.choice(n // 2, width - 1, replace=False))
    col = np.sort((np.arange(n)[:, None] + off) % n, 1)
    val = g.standard_normal((n, width)) + 4.0 * width * (col == np.arange(n)[:, None])
    return CSR(n, width * np.arange(n + 1, dtype=np.int64), col.reshape(-1).astype(np.int32), val.reshape(-1))


def problems(skf, A, basis, m, k, zeta, count):
    op = skf.upload_csr(A.rowptr, A.colind, A.values.astype(np.float32 if basis == torch.float32 else np.float64),
                        device="cuda")
    f = skf.make_func("invsqrt", 0.5 * float(op.csr.norm_inf()))
    probs = []
    for r in range(count):
        b = torch.as_tensor(gaussian_rhs(A.n, 1 + r), device="cuda")
        S = skf.Sketch(skf.SPARSE_SIGN, A.n, 4 * m, zeta, 20 + r)
        probs.append((skf.SGMRES if r % 2 else skf.SFOM, op.csr, S, b, f, skf.make_params(m, k, basis_dtype=basis),
                      torch.full_like(b, float("nan")), skf.new_info()))
    return op, probs


# 4 lanes: N = 20000 takes the middle partition, 40000 and 70001 the last one
# (ragged last slice); from 77825 = 152 x 512 + 1 on a summand is two slices (77857: an
# odd number of slices, the last one ragged); 155648 = 152 x 1024 is the last size of
# the short form and 155649 the first beyond it
@pytest.mark.parametrize("A,basis,k,zeta", [
    (convdiff_2d(200, (60.0, 50.0)), torch.float64, 2, 8), (convdiff_2d(200, (60.0, 50.0)), torch.float32, 2, 8),
    (convdiff_3d(27, (50.0, 50.0, 50.0)), torch.float64, 4, 8), (convdiff_3d(41, (50.0, 50.0, 50.0)), torch.float32, 1, 8),
    (wide(20_000, 12, 1), torch.float64, 2, 8), (wide(70_001, 8, 2), torch.float64, 3, 16),
    (wide(77_857, 5, 5), torch.float64, 2, 8), (wide(155_648, 3, 3), torch.float64, 2, 8),
    (wide(155_649, 3, 4), torch.float32, 2, 8)])
def test_bits_do_not_depend_on_the_lanes(skf, A, basis, k, zeta):
    op, probs = problems(skf, A, basis, 12, k, zeta, 4)
    skf.solve_batched(probs, lanes=4)
    torch.cuda.synchronize()
    for method, csr, S, b, f, p, x, info in probs:
        xi, ii = torch.empty_like(b), skf.new_info()
        skf.solve(method, csr, S, b, f, p, x=xi, info=ii)
        assert skf.read_info(ii)["status"] == 0
        assert torch.equal(x, xi) and torch.equal(info, ii)


@pytest.mark.parametrize("N,width,k", [(155_648, 3, 2), (155_649, 3, 4), (116_737, 8, 3), (77_824, 5, 4), (77_825, 5, 2),
                                       (40_000, 12, 1)])
def test_columns_at_the_edges_of_the_short_form(skf, N, width, k):
    """Against the FP64 oracle, 1e-11 per column (as elsewhere)."""
    A, m = wide(N, width, N), 6
    op = upload(skf, A)
    b = gaussian_rhs(N, 3)
    S = skf.Sketch(skf.SPARSE_SIGN, N, 32, 8, 13)
    with skf.arnoldi_mode(skf.ARNOLDI_PERSISTENT):
        V, vs, SV, SAV, H = skf.arnoldi_trunc(op.csr, S, torch.as_tensor(b, device="cuda"), m, k)
    torch.cuda.synchronize()
    ar = o_arnoldi(csr_to_scipy(A), b, m, k, OSketch("sparse_sign", N, 32, 8, 13))
    Vn = (V * vs[:, None]).cpu().numpy()
    for j in range(m):
        assert rel(Vn[j], ar["V"][:, j]) < 1e-11, j
        assert rel(SV[j].cpu().numpy(), ar["SV"][:, j]) < 1e-11, j
        assert rel(SAV[j].cpu().numpy(), ar["SAV"][:, j]) < 1e-11, j


def test_lanes_of_small_solves_overlap(skf):
    """16 solves of 25600 rows: 34 CTAs each on 8 lanes (of 304 that fit), so all
    lanes run at once; a third of that overlap is asked for."""
    op, probs = problems(skf, convdiff_2d(160, (60.0, 50.0)), torch.float64, 40, 2, 8, 16)

    def timed(lanes):
        ms = []
        for _ in range(6):
            t0, t1 = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            t0.record()
            skf.solve_batched(probs, lanes=lanes)
            t1.record()
            torch.cuda.synchronize()
            ms.append(t0.elapsed_time(t1))
        return min(ms[2:])

    assert timed(1) / timed(8) > 8 / 3
