"""The separable boundaries at the edges of their size rules, through the
cluster environments they close, against the FP64 oracle (tolerance as in
test_gpu_parity: 1e-10 on expectation values)."""
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


# one entry per pair (D = 1); one CTA per side (D = 2, 4); a cluster with more
# CTAs than some have pairs (D = 5) and with more pairs than lanes (D = 8);
# beyond the packed path (D = 9); single rows and columns
@pytest.mark.parametrize("Ly,Lx,D,n", [(3, 4, 1, 2), (5, 2, 2, 1), (4, 5, 4, 2), (3, 3, 5, 2), (3, 3, 8, 1),
                                       (2, 3, 9, 1), (1, 6, 3, 2), (6, 1, 3, 2)])
def test_cluster_environments_at_cu0_edges(peps, Ly, Lx, D, n):
    from paper_1311_6696_gb300 import synth
    A = synth.peps_gauss(Ly, Lx, 2, D, seed=60 + D)
    got = peps.env_cluster(A, n, chi=D * D, mode="var")
    want = O.env_cluster(A, n, chi=D * D, mode="var")
    for kind, op in (("site", O.SZ), ("hbond", O.SDOTS), ("vbond", O.SDOTS)):
        if kind != "site" and (n == 1 or (Lx if kind == "hbond" else Ly) == 1):
            continue
        g, w = got.expect(kind, op).ravel(), np.asarray(O.expect_all(want, kind, op), dtype=float).ravel()
        assert np.max(np.abs(g - w) / np.maximum(np.abs(w), 1e-2)) < 1e-10, kind


# Rows too long for shared memory beside columns of one or two sites: all four
# sides take the kernel that the long ones need.
@pytest.mark.parametrize("Ly,Lx,D", [(1, 2600, 2), (2570, 1, 2), (1, 1300, 3), (1, 800, 4)])
def test_long_thin_lattices(peps, Ly, Lx, D):
    from paper_1311_6696_gb300 import synth
    A = synth.peps_gauss(Ly, Lx, 2, D, seed=60 + D)
    got = peps.env_cluster(A, 1, chi=D * D, mode="var").expect("site", O.SZ).ravel()
    want = np.asarray(O.expect_all(O.env_cluster(A, 1, chi=D * D, mode="var"), "site", O.SZ), dtype=float).ravel()
    assert np.max(np.abs(got - want) / np.maximum(np.abs(want), 1e-2)) < 1e-10
