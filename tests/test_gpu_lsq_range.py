"""Least squares (Alg. 12) over the range of its right-hand side: b is FP64, and
the solution for b scaled by s is s times the solution for b, found in as many
iterations, whatever s is -- on every form of the pass over A."""
import numpy as np
import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu


def problem(n, d, csr):
    import paper_2203_02798_gb300 as lsk
    rng = np.random.default_rng(n + d)
    if not csr:
        return torch.from_numpy(workloads.dense_normal(n, d, seed=n + d)).cuda(), rng.standard_normal(n)
    V, J, I = workloads.csr_bernoulli(n, d, 0.1, seed=n + d)
    return lsk.csr_from_numpy(V, J, I, d), rng.standard_normal(n)


@pytest.mark.parametrize("scale", [1e-30, 1e-20, 1e-12, 1e18, 1e20])
@pytest.mark.parametrize("n,d,csr", [(20_000, 32, False), (9001, 127, False), (9000, 256, False), (4000, 300, False),
                                     (20_000, 32, True), (9000, 256, True)])
def test_scaled_right_hand_side(n, d, csr, scale):
    import paper_2203_02798_gb300 as lsk
    A, b = problem(n, d, csr)
    x0, info0 = lsk.sketch_precondition_lsq(A, torch.from_numpy(b).cuda())
    x, info = lsk.sketch_precondition_lsq(A, torch.from_numpy(scale * b).cuda())
    # both stop at eta <= 1e-10 with cond(A) below 10: they agree to 1e-9
    assert info["eta"] <= 1e-10 and info["refinements"] <= info0["refinements"] + 1
    assert abs(info["iters"] - info0["iters"]) <= 0.1 * info0["iters"] + 2
    assert torch.linalg.norm(x / scale - x0) <= 1e-9 * torch.linalg.norm(x0)


@pytest.mark.parametrize("scale", [1e-100, 1e-42, 1e40, 1e100])
@pytest.mark.parametrize("n,d,csr", [(20_000, 32, False), (9001, 127, False), (9000, 256, False), (4000, 300, False),
                                     (20_000, 32, True), (9000, 256, True)])
def test_right_hand_side_beyond_fp32(n, d, csr, scale):
    """b, x and A^T b outside FP32's range: everything but the inner solve's
    products is FP64, here and in Alg. 10."""
    import paper_2203_02798_gb300 as lsk
    A, b = problem(n, d, csr)
    b0, b1 = torch.from_numpy(b).cuda(), torch.from_numpy(scale * b).cuda()
    for solve in (lambda v: lsk.sketch_precondition_lsq(A, v)[0], lambda v: lsk.least_squares_gram(A, v, refine=2)):
        x0 = solve(b0)
        assert torch.linalg.norm(solve(b1) / scale - x0) <= 1e-9 * torch.linalg.norm(x0)


@pytest.mark.parametrize("n,d", [(20_000, 32), (20_000, 64), (20_000, 100), (20_001, 127), (30_000, 256)])
def test_residual_keeps_64_bits(n, d):
    """Alg. 10 refined on b = A x: x comes back to 64 bits.  b is A x rounded
    (2^-53 of a row), the residual rounds as much, x itself 2^-53, and cond(A)
    is below 1.25: 4 of them bound the error.  A residual of 48 bits leaves
    2^-49 of each entry of x (1e-15 in the norm)."""
    import paper_2203_02798_gb300 as lsk
    A = workloads.dense_normal(n, d, seed=3)
    xt = np.random.default_rng(d).standard_normal(d)
    b = (A.astype(np.longdouble) @ xt.astype(np.longdouble)).astype(np.float64)
    x = lsk.least_squares_gram(torch.from_numpy(A).cuda(), torch.from_numpy(b).cuda(), refine=4).cpu().numpy()
    assert np.linalg.norm(x - xt) <= 4 * 2.0 ** -53 * np.linalg.norm(xt)


def test_conversion_of_every_kind_of_entry():
    """Entries of A that are zero, subnormal or near the ends of FP32's range
    reach the residual exactly: one refined solve with a diagonal A."""
    import paper_2203_02798_gb300 as lsk
    v = np.array([1.0, 2.0 ** -60, 2.0 ** 60, 1.0 + 2.0 ** -23, 3.0 * 2.0 ** -61, -(2.0 ** 59)], dtype=np.float32)
    d, n = v.size, 64
    A = np.zeros((n, d), dtype=np.float32)
    A[np.arange(d), np.arange(d)] = v
    A[20, 0] = 1e-41                      # subnormal, times x_0 = 2^70: part of b's row 20
    xt = np.array([2.0 ** 70, 3.0, 5.0, -7.0, 1.5, 0.25])
    b = (A.astype(np.longdouble) @ xt.astype(np.longdouble)).astype(np.float64)
    x = lsk.least_squares_gram(torch.from_numpy(A).cuda(), torch.from_numpy(b).cuda(), refine=4).cpu().numpy()
    assert np.all(np.abs(x - xt) <= 4 * 2.0 ** -53 * np.abs(xt))
