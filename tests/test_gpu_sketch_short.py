"""Sketch apply around the length up to which one CTA takes the maximum of a
column and the keys are not cleared: exact sums as elsewhere (1e-14), and a
zero column stays zero after a call that left other keys behind."""
import numpy as np
import pytest
import torch

from oracle.sketch import Sketch as OSketch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N", [1, 255, 8192, 8193])
@pytest.mark.parametrize("noalloc", [False, True])
def test_short_columns(skf, N, noalloc):
    apply = skf.sketch_apply_noalloc if noalloc else skf.sketch_apply
    S = skf.Sketch(skf.SPARSE_SIGN, N, 100, 8, 21)
    O = OSketch("sparse_sign", N, 100, 8, 21)
    g = np.random.default_rng(N)
    for scale in (1e30, 1.0):
        X = g.standard_normal((N, 3)) * scale
        X[:, 1] = 0.0
        got = apply(S, torch.as_tensor(X, device="cuda")).cpu().numpy()
        want = O @ X
        assert not got[:, 1].any()
        for c in (0, 2):
            assert np.linalg.norm(got[:, c] - want[:, c]) <= 1e-14 * np.linalg.norm(want[:, c])


# stripes of 64 / 65 rows (8 / 4 copies of the bins by lane) and of 128 / 129 (4 / the
# general pattern, one)
@pytest.mark.parametrize("s", [512, 520, 1024, 1032])
def test_bin_copies_at_the_stripe_widths(skf, s):
    N = 20_011
    X = np.random.default_rng(s).standard_normal((N, 3))
    S = skf.Sketch(skf.SPARSE_SIGN, N, s, 8, 21)
    got = skf.sketch_apply(S, torch.as_tensor(X, device="cuda")).cpu().numpy()
    want = OSketch("sparse_sign", N, s, 8, 21) @ X
    for c in range(3):
        assert np.linalg.norm(got[:, c] - want[:, c]) <= 1e-14 * np.linalg.norm(want[:, c])
