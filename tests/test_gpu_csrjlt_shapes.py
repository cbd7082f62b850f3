"""csrjlt (Alg. 4) at the edges of its blocks: rows of G just below, at and
past a block, one to four of them, rows of A with more nonzeros than a batch,
unsorted and repeated columns, wide A; and the same result twice."""
import numpy as np
import pytest
import torch

import workloads
from oracle import gaussian as oga

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lsk():
    import paper_2203_02798_gb300 as p
    p.load_library()
    return p


def shuffled(V, J, I, seed):
    """The entries of each row in another order, the first one repeated with a
    column that is already there."""
    rng = np.random.default_rng(seed)
    V, J = V.copy(), J.copy()
    for a, b in zip(I[:-1], I[1:]):
        o = a + rng.permutation(b - a)
        V[a:b], J[a:b] = V[o], J[o]
        if b - a > 2:
            J[a] = J[a + 1]
    return V, J


@pytest.mark.parametrize("n,d,p,m,prec", [
    (700, 20, 0.3, 1, "fp32"), (700, 33, 0.3, 4, "fp32"), (257, 5, 0.9, 5, "bf16"), (3_000, 64, 0.05, 16, "fp32"),
    (2_049, 200, 0.02, 63, "fp32"), (2_048, 200, 0.02, 64, "fp32"), (2_047, 230, 0.02, 65, "fp32"),
    (1_500, 256, 0.9, 130, "fp32"), (900, 640, 0.5, 70, "bf16"), (600, 1500, 0.4, 33, "fp32")])
def test_csrjlt_shapes(lsk, n, d, p, m, prec):
    V, J, I = workloads.csr_bernoulli(n, d, p, seed=m)
    V, J = shuffled(V, J, I, m)
    op = oga.PREC_BF16 if prec == "bf16" else oga.PREC_FP32
    A = lsk.csr_from_numpy(V, J, I, d)
    C = lsk.csrjlt(A, m, 13, prec)
    again = lsk.csrjlt(A, m, 13, prec)
    lsk.context().sync()
    assert torch.equal(C, again)
    dense = np.zeros((n, d))
    mag = np.zeros((n, d))
    rows = np.repeat(np.arange(n), np.diff(I))
    np.add.at(dense, (rows, J), V.astype(np.float64))
    np.add.at(mag, (rows, J), np.abs(V).astype(np.float64))
    G = oga.gaussian_columns(m, 0, n, 13, op, oga.STREAM_JLT)
    # FP32 products and sums of a column's nonzeros, G's entries within a few
    # ulp (bf16: the odd entry rounded to the other neighbour)
    bound = (2.0**-21 if prec == "fp32" else 2.0**-12) * (np.abs(G) @ mag) * np.sqrt((mag != 0).sum(0)[None, :] + 8)
    assert np.all(np.abs(C.cpu().numpy() - G @ dense) <= bound + 1e-30)


def test_csrjlt_bad_rows_are_reported(lsk):
    V, J, I = workloads.csr_bernoulli(2_000, 30, 0.1, seed=3)
    bad = J.copy()
    bad[777] = 30                                       # a column past d: skipped and reported
    lsk.csrjlt(lsk.csr_from_numpy(V, bad, I, 30), 20, 1)
    with pytest.raises(lsk.LskError, match="BAD_CSR"):
        lsk.context().sync()
    C = lsk.csrjlt(lsk.csr_from_numpy(V, J, I, 30), 20, 1)
    lsk.context().sync()
    assert torch.isfinite(C).all()
