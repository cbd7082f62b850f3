"""CSR: the CountSketch by reductions and the Gram matrix by reductions, at the
edges of the rules that choose them and of their groups of 32 rows."""
import numpy as np
import pytest
import torch

from oracle import countsketch as ocs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lsk():
    import paper_2203_02798_gb300 as p
    p.load_library()
    return p


def integers(counts, d, seed):
    """Rows with the given numbers of nonzeros, unsorted and repeated columns
    among them, whole numbers: sums are exact in FP32 in any order."""
    rng = np.random.default_rng(seed)
    I = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    J = rng.integers(0, d, size=I[-1]).astype(np.int32)
    V = rng.integers(-4, 5, size=I[-1]).astype(np.float32)
    return V, J, I


def counts_of(kind, n):
    c = np.random.default_rng(n).integers(0, 4, size=n)
    if kind == "long":        # rows longer than a warp's batch among empty ones
        c[:] = 0
        c[::37] = 301
        c[n // 2] = 5000
    elif kind == "dense":     # more than four a row
        c[:] = 40
    return c


def csr(lsk, V, J, I, n, d):
    return lsk.CSR(torch.from_numpy(V).cuda(), torch.from_numpy(J).cuda(), torch.from_numpy(I).cuda(), n, d)


def dense(V, J, I, n, d):
    A = np.zeros((n, d))
    np.add.at(A, (np.repeat(np.arange(n), np.diff(I)), J), V)
    return A


@pytest.mark.parametrize("kind", ["sparse", "long", "dense"])
@pytest.mark.parametrize("n,d,r", [(1, 40, 500), (31, 40, 500), (32, 129, 127), (33, 128, 128), (1000, 7, 3000),
                                   (5000, 64, 255), (5000, 64, 256), (4000, 300, 100)])
def test_csr_countsketch_is_exact(lsk, kind, n, d, r):
    V, J, I = integers(counts_of(kind, n), d, n + r)
    bucket, sign = ocs.countsketch_hash(n, r, 5)
    ref = np.zeros((r, d))
    np.add.at(ref, bucket, dense(V, J, I, n, d) * sign[:, None])
    A = csr(lsk, V, J, I, n, d)
    assert np.array_equal(lsk.cs_sketch(A, r, 5).cpu().numpy(), ref)
    SA = lsk.cs_sketch(A, r, 5)
    lsk.sketch_rows(A, r, 0, 5, out=SA, accumulate=True)
    assert np.array_equal(SA.cpu().numpy(), 2 * ref)


@pytest.mark.parametrize("kind", ["sparse", "long", "dense"])
@pytest.mark.parametrize("n,d", [(1, 5), (31, 40), (33, 221), (5000, 222), (6000, 64), (3000, 700)])
def test_csr_gram_is_exact(lsk, kind, n, d):
    V, J, I = integers(counts_of(kind, n), d, n + d)
    A = dense(V, J, I, n, d)
    assert np.array_equal(lsk.gram(csr(lsk, V, J, I, n, d)).cpu().numpy(), A.T @ A)


@pytest.mark.parametrize("spoil", ["column", "pointer"])
def test_bad_csr_is_reported(lsk, spoil):
    """A column past the last and a row pointer past the entries are skipped and
    reported; the other rows still count."""
    n, d, r = 200, 64, 1024
    V, J, I = integers(counts_of("sparse", n), d, 1)
    if spoil == "column":
        J[0] = d
    else:
        I = I.copy()
        I[100] = len(V) + 7
    A = csr(lsk, V, J, I, n, d)
    for call in (lambda: lsk.cs_sketch(A, r, 5), lambda: lsk.gram(A)):
        call()
        with pytest.raises(lsk.LskError) as ei:
            lsk.context().sync()
        assert ei.value.name == "BAD_CSR"


@pytest.mark.parametrize("kind", ["sparse", "long", "dense"])
@pytest.mark.parametrize("n,d", [(1, 5), (31, 40), (33, 64), (5000, 64), (600, 700)])
def test_csr_row_norms(lsk, kind, n, d):
    """||a_i B||^2 = a_i (B B^T) a_i^T for whole numbers: every product and sum of
    the quadratic form is exact in FP32 below 2^24, so the result is."""
    counts = np.minimum(counts_of(kind, n), 60 if kind == "dense" else 301)
    V, J, I = integers(counts, d, n + d)
    V = np.sign(V).astype(np.float32)
    B = np.random.default_rng(d).integers(-1, 2, size=(d, 3)).astype(np.float32)
    ref = np.square(dense(V, J, I, n, d) @ B).sum(1)
    got = lsk.rownorms_prod(csr(lsk, V, J, I, n, d), torch.from_numpy(B).cuda()).cpu().numpy()
    assert np.array_equal(got, ref)
