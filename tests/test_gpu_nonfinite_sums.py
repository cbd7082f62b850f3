"""Sums of partials that are not finite, or leave FP32's range on their way, come
out as sums in 64 bits do: an infinity stays one, NaN appears only where
infinities of both signs meet, and alpha can bring a large sum back."""
import numpy as np
import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu


def same(got, want):
    """Infinities, signs and NaNs where 64-bit sums have them; the rest finite and close."""
    want = want.astype(np.float32)
    assert np.array_equal(np.isnan(got), np.isnan(want)) and np.array_equal(np.isinf(got), np.isinf(want))
    assert np.array_equal(got[np.isinf(want)], want[np.isinf(want)])
    ok = np.isfinite(want)
    assert np.allclose(got[ok], want[ok], rtol=1e-4, atol=1e-4 * np.abs(want[ok]).max())


def sparse(n, d, density, seed):
    """CSR arrays with two positive infinities in column 3, and one of each sign in column 5."""
    V, J, I = workloads.csr_bernoulli(n, d, density, seed=seed)
    in3, in5 = np.flatnonzero(J == 3), np.flatnonzero(J == 5)
    V[in3[[2, 40]]] = np.inf
    V[in5[7]], V[in5[60]] = np.inf, -np.inf
    A = np.zeros((n, d))
    np.add.at(A, (np.repeat(np.arange(n), np.diff(I)), J), V)
    return V, J, I, A


@pytest.mark.parametrize("n,d,density", [(20_000, 40, 0.05), (9000, 64, 0.25), (6000, 300, 0.02)])
def test_csr_gram(n, d, density):
    import paper_2203_02798_gb300 as lsk
    V, J, I, A = sparse(n, d, density, seed=1)
    with np.errstate(invalid="ignore"):
        rows = np.flatnonzero(np.isinf(A).any(axis=1))
        P = A.copy()
        P[rows] = 0.0
        want = P.T @ P
        for i in rows:                     # the products of a row's nonzeros only
            j = np.flatnonzero(A[i])
            want[np.ix_(j, j)] += np.outer(A[i, j], A[i, j])
    same(lsk.gram(lsk.csr_from_numpy(V, J, I, d)).cpu().numpy(), want)


@pytest.mark.parametrize("n,d,m", [(20_000, 40, 16), (9000, 100, 70)])
def test_csrjlt(n, d, m):
    import paper_2203_02798_gb300 as lsk
    V, J, I, A = sparse(n, d, 0.05, seed=2)
    C = lsk.csrjlt(lsk.csr_from_numpy(V, J, I, d), m, 5, "fp32").cpu().numpy()
    one = np.ones((n, 1), dtype=np.float32)            # G's signs at an entry: the sketch of one row
    for col in (3, 5):
        at = np.flatnonzero(np.isinf(A[:, col]))
        signs = []
        for i in at:
            ptr = np.zeros(n + 1, dtype=np.int64)
            ptr[i + 1:] = 1
            g = lsk.csrjlt(lsk.csr_from_numpy(one[i], np.zeros(1, dtype=np.int32), ptr, 1), m, 5, "fp32").cpu().numpy()[:, 0]
            signs.append(np.sign(g) * np.sign(A[i, col]))
        s = np.array(signs)
        want = np.where((s > 0).all(0), np.inf, np.where((s < 0).all(0), -np.inf, np.nan))
        assert np.array_equal(C[:, col], want, equal_nan=True)
    others = [j for j in range(d) if j not in (3, 5)]
    assert np.isfinite(C[:, others]).all()


def test_gaussian_stage():
    import paper_2203_02798_gb300 as lsk
    r, d, k = 3000, 20, 64
    SA = workloads.dense_normal(r, d, seed=4)
    SA[100, 3] = np.inf
    SA[200, 5], SA[2500, 5] = np.inf, -np.inf
    G = lsk.debug_gauss(k, r, 9).cpu().numpy().astype(np.float64)
    with np.errstate(invalid="ignore"):
        want = G @ SA.astype(np.float64)
    same(lsk.gauss_sketch(torch.from_numpy(SA).cuda(), k, 9, "fp32").cpu().numpy(), want)


def test_large_sums_and_alpha():
    """Products of 1.6e37, a few to a partial sum, 2.6e39 in all, times alpha = 1e-20."""
    import paper_2203_02798_gb300 as lsk
    n, d = 8000, 50
    V, J, I = np.full(n, 4e18, dtype=np.float32), (np.arange(n) % d).astype(np.int32), np.arange(n + 1, dtype=np.int64)
    C = lsk.gram(lsk.csr_from_numpy(V, J, I, d), alpha=1e-20).cpu().numpy()
    want = np.eye(d) * (n / d) * float(V[0]) ** 2 * 1e-20
    assert np.allclose(C, want, rtol=1e-5, atol=0.0)


@pytest.mark.parametrize("n,d", [(300_000, 32), (200_000, 130)])
def test_large_sums_of_dense_products(n, d):
    """Products of 1e35: a few thousand rows' sums leave FP32's range, no thousand's
    do.  The CUDA cores, which form them, add up 1,024 equal products in FP32 at a
    time, each addition rounding the same way: within 1,024 x 2^-24."""
    import paper_2203_02798_gb300 as lsk
    A = 3e17 * torch.sign(torch.randn((n, d), generator=torch.Generator(device="cuda").manual_seed(3), device="cuda"))
    C = lsk.gram(A, alpha=1e-20, prec="fp32").double()
    want = 1e-20 * (A.double().T @ A.double())
    assert torch.all((C - want).abs() <= 1024 * 2.0 ** -24 * want.diagonal().max())
