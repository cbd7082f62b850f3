"""FP32 Gram matrix on the tensor cores (lsk_gram_prec FP32, dense, d <= 256):
edges of its 128-column panels and 32-row chunks, strided and unaligned rows,
and the inputs it leaves to the CUDA-core kernel."""
import numpy as np
import pytest

import workloads
from oracle import gram as ogr

pytestmark = pytest.mark.gpu
U24 = 2.0**-24


@pytest.fixture(scope="module")
def lsk():
    import paper_2203_02798_gb300 as m
    m.load_library()
    return m


def gram(lsk, A, ld=None, **kw):
    import torch
    n, d = A.shape
    buf = torch.zeros((n, ld or d), dtype=torch.float32, device="cuda")
    buf[:, :d] = torch.from_numpy(A)
    C = lsk.gram(buf[:, :d], prec="fp32", **kw)
    lsk.context().sync()
    return C.cpu().numpy().astype(np.float64)


# one and two panels, a panel of one column, ragged rows (a last chunk of one
# row), rows that are not 16-byte aligned, a row stride, few and many segments
@pytest.mark.parametrize("n,d,ld", [(16_384, 32, None), (40_001, 33, None), (8_193, 64, 72), (8_192, 127, 129),
                                    (4_097, 128, None), (4_100, 129, None), (30_000, 160, 161), (2_080, 256, None),
                                    (250_003, 200, None), (400_000, 100, None)])
@pytest.mark.parametrize("shape", ["normal", "scaled", "outliers", "offset"])
def test_gram_fp32_tensor_cores(lsk, n, d, ld, shape):
    """Per entry: the result is stored in FP32 (2^-24 of |C|), each entry of A is
    kept to 2^-24 of its column's largest recent entry, and a CTA's few segment
    sums are rounded to nearest: within 4 x 2^-24 of sqrt(C_aa C_bb) in all."""
    A = workloads.dense_normal(n, d, seed=d)
    if shape == "scaled":
        A *= (10.0 ** np.linspace(-3, 3, d)).astype(np.float32)
    elif shape == "outliers":
        A[:5] *= 100.0
    elif shape == "offset":
        A = (1.0 + 0.01 * A).astype(np.float32)
    C = gram(lsk, A, ld)
    ref = ogr.gram_dense(A.astype(np.float64))
    g = np.sqrt(np.diag(ref))
    assert np.all(np.abs(C - ref) <= 4 * U24 * np.outer(g, g))
    assert np.array_equal(C, C.T)


def test_gram_fp32_alpha_beta(lsk):
    import torch
    A = workloads.dense_normal(20_000, 140, seed=1)
    C0 = workloads.dense_normal(140, 140, seed=2)
    got = gram(lsk, A, alpha=0.5, beta=-2.0, C=torch.from_numpy(C0).cuda())
    ref = ogr.gram_dense(A.astype(np.float64), 0.5, -2.0, C0.astype(np.float64))
    assert np.linalg.norm(got - ref) <= 4 * U24 * np.linalg.norm(ref)


@pytest.mark.parametrize("value", [np.nan, np.inf, 1e25])
def test_gram_fp32_outside_the_split(lsk, value):
    """An entry that is not finite (or whose square is not) reaches exactly the
    row and column of C it belongs to, as FP32 arithmetic has it, and beta's C
    is read once."""
    import torch
    A = workloads.dense_normal(20_000, 70, seed=3)
    A[12_345, 7] = value
    C0 = torch.ones((70, 70), dtype=torch.float32, device="cuda")
    got = gram(lsk, A, beta=1.0, C=C0)
    ok = np.ones(70, dtype=bool)
    ok[7] = False
    ref = ogr.gram_dense(A[:, ok].astype(np.float64)) + 1.0
    assert np.linalg.norm(got[np.ix_(ok, ok)] - ref) <= 1e-6 * np.linalg.norm(ref)
    assert not np.isfinite(got[7, 7])
    if np.isnan(value):
        assert np.all(np.isnan(got[7])) and np.all(np.isnan(got[:, 7]))


def test_gram_fp32_small_magnitudes(lsk):
    A = workloads.dense_normal(20_000, 70, seed=4)
    A[:, :20] *= np.float32(1e-17)      # products near the bottom of FP32's range
    got = gram(lsk, A)
    ref = ogr.gram_dense(A.astype(np.float64))
    g = np.sqrt(np.diag(ref))
    assert np.all(np.abs(got - ref) <= 1e-5 * np.outer(g, g))
