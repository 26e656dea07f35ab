"""The FP64 factorisations and contractions at the edges of their size rules,
through the norm sweep against the FP64 oracle (tolerance as in test_gpu_parity: 1e-10 absolute
on ln N)."""
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


# Shapes of the QR's boundary tensors, rows x columns: one CTA (12x3), ragged
# rows over a cluster (175x7), more columns than four threads each cover and a
# triangle in global memory (1620x180), tall-skinny candidates (1188x33).  The
# next three are for the contractions: one-element groups and K below a tile
# (D = 1, chi = 1), ragged tiles with K split over a cluster (D = 7, chi = 5).
# The last are for the SVD: fewer columns than its preconditioning takes (9),
# wider than high and higher than wide (27x81, 81x27), odd widths (49).
@pytest.mark.parametrize("Ly,Lx,D,chi,mode", [(4, 6, 2, 3, "var"), (4, 4, 5, 7, "var"), (4, 5, 3, 20, "svd"),
                                              (4, 4, 6, 33, "var"), (3, 5, 1, 4, "var"),
                                              (4, 3, 3, 1, "var"), (4, 4, 7, 5, "var"),
                                              (4, 4, 3, 1, "svd"), (3, 5, 3, 9, "svd"), (3, 4, 7, 7, "svd")])
def test_norm_at_factor_edges(peps, Ly, Lx, D, chi, mode):
    from paper_1311_6696_gb300 import synth
    A = synth.peps_gauss(Ly, Lx, 2, D, seed=40 + D)
    got, want = peps.norm(A, chi, mode=mode, seed=2), O.norm(A, chi=chi, mode=mode, seed=2)
    assert abs(got[0] - want[0]) < 1e-10 and got[1] == want[1]


# Boundary tensors of 1024 rows and more, whose QR is split over every SM:
# rows and columns that are no multiple of a warp's or a CTA's share
# (1500x60), and more of them than four threads each cover (2240x140); just
# below the rule, on one cluster (1008x63).  |ln N| is a few tens, and both
# sides round in FP64 only: the 1e-10 above.
@pytest.mark.parametrize("Ly,Lx,D,chi", [(4, 6, 5, 60), (4, 6, 4, 140), (4, 6, 4, 63)])
def test_norm_with_tall_boundaries(peps, Ly, Lx, D, chi):
    from paper_1311_6696_gb300 import synth
    A = synth.peps_gauss(Ly, Lx, 2, D, seed=60 + D)
    got, want = peps.norm(A, chi, mode="var", seed=2), O.norm(A, chi=chi, mode="var", seed=2)
    assert abs(got[0] - want[0]) < 1e-10 and got[1] == want[1]


# Wide factorisations, through svd mode: rows of a square matrix in shared
# memory and the triangular factor's columns beside them in global memory
# (448 columns), everything but the sums in global memory (608 columns, where
# those columns alone would fill the shared memory).
@pytest.mark.parametrize("Ly,Lx,D,chi", [(4, 6, 4, 28), (4, 6, 4, 38)])
def test_norm_with_wide_factorisations(peps, Ly, Lx, D, chi):
    from paper_1311_6696_gb300 import synth
    A = synth.peps_gauss(Ly, Lx, 2, D, seed=80 + D)
    got, want = peps.norm(A, chi, mode="svd"), O.norm(A, chi=chi, mode="svd")
    assert abs(got[0] - want[0]) < 1e-10 and got[1] == want[1]


def test_tall_boundaries_beside_other_work(peps):
    """The CTAs of a QR on every SM wait for one another: with the device busy
    on another stream when it is launched, the norm is the same to the bit."""
    import torch
    from paper_1311_6696_gb300 import synth
    A = synth.peps_gauss(4, 6, 2, 5, seed=65)
    alone = peps.norm(A, 60, mode="var", seed=2)
    x = torch.randn(4096, 4096, device="cuda", dtype=torch.float64)
    torch.cuda.synchronize()
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        for _ in range(8):
            y = x @ x
    assert peps.norm(A, 60, mode="var", seed=2) == alone
    side.synchronize()
    assert torch.equal(y, x @ x)
