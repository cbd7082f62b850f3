"""Grouped CountSketch preparation and Gaussian slices at the edges of their rules."""
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


# (n, d, r): rows ranked in shared memory (r <= 4096 and n >= 2r) and one short of
# either condition; a block's run of 8,192 rows less one, full and one over;
# compacted sketches (n < 4r) with one bucket more than a round of the compaction
SHAPES = [(8191, 32, 1024), (8192, 32, 1024), (8193, 32, 1024), (2047, 32, 1024), (2048, 32, 1024),
          (8192, 64, 4096), (8200, 64, 4097), (40_000, 64, 4097), (70_000, 16, 64), (300, 20, 8193), (4100, 24, 8192)]


def test_grouped_preparation_edges(lsk):
    """Each problem's scores agree with its own pipeline's: BF16 draws are the
    same in both, so the difference is FP32 rounding of sums of at most 70,000
    terms in another order: 2^-24 sqrt(70000) = 1.6e-5 in a sketch entry's norm
    at worst, doubled by the square of the norms."""
    probs = [(torch.from_numpy(workloads.dense_normal(n, d, seed=i)).cuda(), r, 4 * d, 40 + i)
             for i, (n, d, r) in enumerate(SHAPES)]
    grouped = lsk.batch_leverage_scores(probs, prec="bf16")
    single = lsk.batch_leverage_scores(probs, prec="bf16", per_problem=True)
    lsk.context().sync()
    for (n, d, r), a, b in zip(SHAPES, grouped, single):
        a, b = a.cpu().numpy().astype(np.float64), b.cpu().numpy().astype(np.float64)
        assert np.linalg.norm(a - b) <= 4e-5 * np.linalg.norm(b), (n, d, r)
