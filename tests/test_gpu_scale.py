"""Site tensors multiplied by a power of two: ln N shifts by its logarithm and
expectation values do not move.  A power of two scales every FP64 product,
sum and factorisation exactly, so what is left is the rounding of the
logarithms: |ln N| stays below 2000 and sums fewer than 100 terms,
100 x 2000 x 1.1e-16 = 2e-11 of ln N; 1e-12 on expectation values."""
import math

import numpy as np
import pytest

from oracle import peps_oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def peps():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_1311_6696_gb300 import peps as P
    return P


def _lattice(Ly, Lx, D, seed):
    """N(0,1) entries with a bond spectrum 1/(1+k) on every leg, unit norm."""
    A = np.random.default_rng(seed).normal(size=(Ly, Lx, 2, D, D, D, D))
    for leg in range(4):
        A *= (1.0 / (1.0 + np.arange(D))).reshape([-1 if k == 3 + leg else 1 for k in range(7)])
    A[0, :, :, 1:] = 0.0
    A[:, 0, :, :, 1:] = 0.0
    A[-1, :, :, :, :, 1:] = 0.0
    A[:, -1, :, :, :, :, 1:] = 0.0
    return A / np.sqrt((A ** 2).sum(axis=tuple(range(2, 7)), keepdims=True))


# The separable boundaries are defined up to a factor.  One-site windows keep
# the rest of the call within range: their environments scale by 2^(-2 k).
@pytest.mark.parametrize("D", [2, 5])
@pytest.mark.parametrize("k", [60, 140, -140])
def test_separable_boundaries_do_not_depend_on_the_scale(peps, D, k):
    A = _lattice(4, 5, D, seed=80 + D)
    a = peps.env_cluster(A, 1, chi=D * D, mode="var")
    b = peps.env_cluster(A * 2.0 ** -k, 1, chi=D * D, mode="var")
    assert np.max(np.abs(a.expect("site", O.SZ) - b.expect("site", O.SZ))) < 1e-12


# A row of 6 sites scales by 2^(-12 k), to 1e-137 (and to 1e137) before it is
# rescaled; fewer columns than the SVD's preconditioning takes (D = 2, chi = 2),
# more of them (D = 3), and the variational fit, whose local tensors carry the
# row's scale as well.
@pytest.mark.parametrize("D,chi,mode", [(2, 2, "svd"), (3, 4, "svd"), (3, 6, "var")])
@pytest.mark.parametrize("k", [10, 22, 38, -38])
def test_full_environments_do_not_depend_on_the_scale(peps, D, chi, mode, k):
    Ly, Lx = 4, 6
    A = _lattice(Ly, Lx, D, seed=70 + D)
    B = A * 2.0 ** -k
    shift = -2.0 * k * math.log(2.0) * Ly * Lx
    ln, sign = peps.norm(A, chi, mode=mode, seed=2)
    ln_b, sign_b = peps.norm(B, chi, mode=mode, seed=2)
    assert abs(ln_b - ln - shift) < 1e-10 and sign_b == sign
    a, b = peps.env_full(A, chi, mode=mode, seed=2), peps.env_full(B, chi, mode=mode, seed=2)
    for kind, op in (("site", O.SZ), ("hbond", O.SDOTS), ("vbond", O.SDOTS)):
        assert np.max(np.abs(a.expect(kind, op) - b.expect(kind, op))) < 1e-12, kind


# Rows down to 1e-148: the local tensors' smaller columns lie below the square
# root of the smallest double, their QR's squares beyond its range.
@pytest.mark.parametrize("D,chi,mode", [(2, 2, "svd"), (3, 4, "svd"), (3, 6, "var"), (4, 5, "var")])
def test_norm_near_the_end_of_the_range(peps, D, chi, mode):
    Ly, Lx, k = 3, 6, 41
    A = _lattice(Ly, Lx, D, seed=90 + D)
    ln, sign = peps.norm(A, chi, mode=mode, seed=2)
    ln_b, sign_b = peps.norm(A * 2.0 ** -k, chi, mode=mode, seed=2)
    assert abs(ln_b - ln + 2.0 * k * math.log(2.0) * Ly * Lx) < 1e-10 and sign_b == sign
