"""Operators on few diagonals: the diagonal copy of the step kernels and the
slices it is an alternative to, at the edges of the rule that chooses (number
of diagonals, row order, filled share, ragged sizes).  FP64 columns against the
oracle at 1e-11 per column, reduced precision against the sketches of the
stored basis (both tolerances as for the same quantities elsewhere)."""
import numpy as np
import pytest

from workloads import gaussian_rhs
from workloads.operators import CSR
from test_gpu_lowprec import arnoldi_lp, check_sketches
from test_gpu_step_edges import check_columns

pytestmark = pytest.mark.gpu

OFFSETS = {
    "one": [0],                                             # mostly unused value slots: slices in FP64
    "tridiagonal": [-1, 0, 1],
    "five_uneven": [-17, -1, 0, 2, 23],
    "six": [-30, -2, -1, 0, 1, 40],                         # seven value slots, one never present
    "seven_upper": [0, 1, 2, 3, 31, 32, 33],
    "eight": [-33, -32, -31, -1, 0, 1, 5, 64],
    "nine": [-40, -33, -2, -1, 0, 1, 2, 33, 40],            # one too many: slices
    "far": [-1000, -1, 0, 1, 1000],                         # outer diagonals mostly or wholly outside
}


def banded(n, offsets, keep=1.0, order="ascending", seed=5):
    """Random entries on the given diagonals (each kept with probability `keep`,
    the main diagonal always, at most eight entries in a row)."""
    rng = np.random.default_rng(seed)
    rowptr, col, val = [0], [], []
    for r in range(n):
        c = [r + o for o in offsets if 0 <= r + o < n and (o == 0 or rng.random() < keep)]
        if len(c) > 8:
            c.pop(rng.integers(4))   # (left of the main diagonal)
        if order == "descending" and r % 7 == 3:
            c = c[::-1]
        if order == "duplicate" and r % 7 == 3 and len(c) < 8:
            c = c + [c[-1]]
        col += c
        val += [3.0 + 0.1 * rng.standard_normal() if q == r else 0.4 * rng.standard_normal() for q in c]
        rowptr.append(len(col))
    return CSR(n, np.array(rowptr, dtype=np.int64), np.array(col, dtype=np.int32), np.array(val))


# one ragged slice, several, a ragged last CTA; from 16384 rows on the copy is
# built: a last slice of one row
# ("one" is not among them: on a diagonal of 3 +- 0.1 each FP64 column magnifies
# the rounding of the one before 30-fold, whatever the kernel)
@pytest.mark.parametrize("n", [29, 5185, 16385])
@pytest.mark.parametrize("name", sorted(set(OFFSETS) - {"one"}))
@pytest.mark.parametrize("form,k", [("persistent", 2), ("persistent", 4), ("two_kernel", 2), ("two_kernel", 3),
                                    ("two_kernel", 6)])
def test_columns(skf, n, name, form, k):
    A = banded(n, OFFSETS[name])
    mode = skf.ARNOLDI_PERSISTENT if form == "persistent" else skf.ARNOLDI_TWO_KERNEL
    check_columns(skf, A, gaussian_rhs(n, 3), 6, k, 24, mode, zeta=7 if n < 64 else 8)


@pytest.mark.parametrize("keep", [0.2, 0.9])
@pytest.mark.parametrize("order", ["ascending", "descending", "duplicate"])
@pytest.mark.parametrize("form", ["persistent", "two_kernel"])
def test_partly_filled_and_unordered_rows(skf, keep, order, form):
    A = banded(17000, OFFSETS["five_uneven"], keep, order)
    mode = skf.ARNOLDI_PERSISTENT if form == "persistent" else skf.ARNOLDI_TWO_KERNEL
    check_columns(skf, A, gaussian_rhs(A.n, 3), 6, 2, 24, mode)


@pytest.mark.parametrize("n", [333, 16385])
@pytest.mark.parametrize("name", sorted(OFFSETS))
@pytest.mark.parametrize("basis,form", [("f32", "persistent"), ("f32", "two_kernel"), ("bf16", "two_kernel")])
def test_reduced_precision_sketches(skf, n, name, basis, form):
    A = banded(n, OFFSETS[name], 0.95)
    m, s = 6, 24
    with skf.arnoldi_mode(skf.ARNOLDI_TWO_KERNEL if form == "two_kernel" else skf.ARNOLDI_AUTO):
        V, SV, SAV, H, info = arnoldi_lp(skf, A, gaussian_rhs(n, 3), m, 2, s, basis)
    assert info["m_eff"] == m
    check_sketches(A, V, SV, SAV, 2, s, m)


# more slices per CTA than warps (several passes of the persistent kernel's loop)
@pytest.mark.parametrize("name", ["six", "eight"])
def test_many_slices_per_cta(skf, name):
    A = banded(100_003, OFFSETS[name], 0.9)
    b = gaussian_rhs(A.n, 3)
    check_columns(skf, A, b, 5, 2, 24, skf.ARNOLDI_PERSISTENT)
    V, SV, SAV, H, info = arnoldi_lp(skf, A, b, 5, 2, 24, "f32")
    assert info["m_eff"] == 5
    check_sketches(A, V, SV, SAV, 2, 24, 5)
