"""Least squares (Alg. 12) at the edges of its passes: each number of lanes a
row and of columns a lane, unaligned rows, fewer rows than a block takes at
once, d beyond the register forms; CSR rows longer than a tile's batch, empty
rows, several runs to a tile, d beyond a pass's shared memory."""
import numpy as np
import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lsk():
    import paper_2203_02798_gb300 as p
    p.load_library()
    return p


def eta(A, b, x):
    """||A^T (b - A x)|| / ||A^T b|| in 64 bits; the call stops at 1e-10."""
    return np.linalg.norm(A.T @ (b - A @ x)) / np.linalg.norm(A.T @ b)


@pytest.mark.parametrize("n,d,pad", [(40, 5, 0), (20_000, 32, 0), (20_001, 33, 0), (3000, 64, 0), (15_000, 100, 0),
                                     (15_000, 100, 1), (9001, 128, 0), (9001, 127, 0), (6000, 200, 4), (5003, 256, 0),
                                     (4000, 255, 0), (3000, 300, 0)])
def test_lsq_dense_shapes(lsk, n, d, pad):
    A = workloads.dense_normal(n, d, seed=n + d)
    b = np.random.default_rng(d).standard_normal(n)
    At = torch.from_numpy(np.hstack([A, A[:, :pad]])).cuda()[:, :d]
    x, info = lsk.sketch_precondition_lsq(At, torch.from_numpy(b).cuda())
    assert info["eta"] <= 1e-10 and eta(A.astype(np.float64), b, x.cpu().numpy()) <= 1e-10


@pytest.mark.parametrize("n,d,kind", [(200, 7, "sparse"), (50_000, 64, "sparse"), (20_000, 256, "sparse"),
                                      (8000, 500, "sparse"), (6000, 100, "long"), (30_000, 40, "gaps")])
def test_lsq_csr_shapes(lsk, n, d, kind):
    rng = np.random.default_rng(n + d)
    counts = rng.integers(1, 9, size=n)
    if kind == "long":
        counts[::50] = 90
    if kind == "gaps":
        counts[5000:9000] = 0
    I = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    J = rng.integers(0, d, size=I[-1]).astype(np.int32)
    V = rng.standard_normal(I[-1]).astype(np.float32)
    b = rng.standard_normal(n)
    A = np.zeros((n, d))
    np.add.at(A, (np.repeat(np.arange(n), counts), J), V)
    At = lsk.CSR(torch.from_numpy(V).cuda(), torch.from_numpy(J).cuda(), torch.from_numpy(I).cuda(), n, d)
    x, info = lsk.sketch_precondition_lsq(At, torch.from_numpy(b).cuda())
    assert info["eta"] <= 1e-10 and eta(A, b, x.cpu().numpy()) <= 1e-10
