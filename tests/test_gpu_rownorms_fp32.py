"""FP32 row norms on the tensor cores (lsk_rownorms_prod FP32, large dense A):
edges of its 32-column chunks and 256-row tiles, general B in one and two
passes, and the rows it hands to the CUDA-core kernel."""
import numpy as np
import pytest
import torch

import workloads
from oracle import rownorms as orn

pytestmark = pytest.mark.gpu
U = 2.0**-24


@pytest.fixture(scope="module")
def lsk():
    import paper_2203_02798_gb300 as m
    m.load_library()
    return m


def check(x, A, B, alpha=1.0, beta_x=0.0):
    """Within the bound of FP32 dot products of length d and FP32 sums of c
    squares."""
    A, B = A.astype(np.float64), B.astype(np.float64)
    y, absy = A @ B, np.abs(A) @ np.abs(B)
    E = (A.shape[1] + 2) * U * absy
    tol = np.sum(2 * np.abs(y) * E + E * E, axis=1) + (B.shape[1] + 2) * U * np.sum(y * y, axis=1)
    want = alpha * orn.rownorms_prod_dense(A, B) + beta_x
    assert np.all(np.abs(x - want) <= abs(alpha) * tol + 4 * U * np.abs(want) + 1e-30)


# d just below, at and past a chunk; c of one accumulator buffer pair and two;
# rows that end inside a tile; strides; a general B that takes two passes
@pytest.mark.parametrize("n,d,c,tri,ld", [
    (1_050_000, 32, 32, True, None), (400_003, 33, 97, False, None), (300_001, 64, 64, True, 68),
    (140_000, 96, 128, False, None), (140_000, 65, 129, False, 67), (70_000, 128, 128, True, None),
    (30_001, 200, 200, False, None), (30_000, 224, 224, True, 225), (20_001, 255, 256, False, None),
    (17_000, 256, 256, False, None), (17_001, 256, 256, True, None)])
def test_rownorms_fp32_tensor_cores(lsk, n, d, c, tri, ld):
    A = workloads.dense_normal(n, d, seed=c) * (10.0 ** np.linspace(-2, 2, d)).astype(np.float32)
    A[:3] *= 100.0
    A[3::50] *= 1e-3                          # far below the typical row: left to the CUDA cores
    A[5::1000] = 0.0
    B = workloads.dense_normal(d, c, seed=d + 1)
    B[:, c // 2] = 0.0
    if tri:
        B = np.triu(B)
    buf = torch.zeros((n, ld or d), dtype=torch.float32, device="cuda")
    buf[:, :d] = torch.from_numpy(A)
    ctx = lsk.context()
    ctx.profile(True)
    ctx.profile_reset()
    x = lsk.rownorms_prod(buf[:, :d], torch.from_numpy(B).cuda(), upper_triangular=tri, prec="fp32")
    ctx.sync()
    names = set(ctx.profile_totals())
    ctx.profile(False)
    assert "rownorm_dense_tc3" in names
    x = x.cpu().numpy().astype(np.float64)
    assert np.all(x[5::1000] == 0.0)
    check(x, A, B)


def test_rownorms_fp32_alpha_beta_and_rows_outside(lsk):
    n, d, c = 60_000, 130, 140
    A, B = workloads.dense_normal(n, d, seed=1), workloads.dense_normal(d, c, seed=2)
    x0 = workloads.dense_normal(n, 1, seed=3)[:, 0]
    A[11] *= np.float32(1e-20)
    A[12] *= np.float32(1e12)
    bad = A.copy()
    bad[13, 5], bad[14, 6] = np.nan, np.inf
    x = torch.from_numpy(x0.copy()).cuda()
    lsk.rownorms_prod(torch.from_numpy(bad).cuda(), torch.from_numpy(B).cuda(), 0.5, -2.0, x, prec="fp32")
    lsk.context().sync()
    got = x.cpu().numpy().astype(np.float64)
    assert np.isnan(got[13]) and not np.isfinite(got[14])
    ok = np.ones(n, dtype=bool)
    ok[[13, 14]] = False
    x64 = x0.astype(np.float64)
    check(got[ok], A[ok], B, 0.5, (-2.0 * x64)[ok])
