"""The CG step of the least-squares solver in every size of cluster that it may
be given: the solution is the one that the largest cluster finds, whether the
factor's rows fit one to a warp (pairs in registers) or not (read in FP64)."""
import numpy as np
import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ctas", [2, 4, 8, 16])
@pytest.mark.parametrize("n,d", [(2000, 5), (5000, 33), (9000, 128), (9000, 129), (12_000, 256), (12_000, 300), (9000, 1024)])
def test_lsq_cluster_sizes(n, d, ctas):
    import paper_2203_02798_gb300 as lsk
    A = workloads.dense_normal(n, d, seed=n + d)
    b = np.random.default_rng(d).standard_normal(n)
    At, bt = torch.from_numpy(A).cuda(), torch.from_numpy(b).cuda()
    r = min(max(d * d, 4 * d), 16_384)
    x0, info0 = lsk.sketch_precondition_lsq(At, bt, r=r)
    ctx = lsk.Context(0)
    lsk.debug_lsq_ctas(ctas, ctx)
    x, info = lsk.sketch_precondition_lsq(At, bt, r=r, ctx=ctx)
    ctx.close()
    # both stop at eta <= 1e-10 and cond(A) is below 10: they agree to 1e-9
    assert info["eta"] <= 1e-10 and abs(info["iters"] - info0["iters"]) <= 4
    assert torch.linalg.norm(x - x0) <= 1e-9 * torch.linalg.norm(x0)
