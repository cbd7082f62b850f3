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
