"""The CountSketch at the edges of its dense gather: each vector width and team
size, whole and shared buckets, empty ones, rows short of a team's batch."""
import numpy as np
import pytest
import torch

import workloads
from oracle import countsketch as ocs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lsk():
    import paper_2203_02798_gb300 as p
    p.load_library()
    return p


def integers(n, d, seed):
    """Entries whose sums are exact in FP32: the result is the same in any order."""
    return np.random.default_rng(seed).integers(-8, 9, size=(n, d)).astype(np.float32)


# (n, d, r): 8, 16 and 32 lanes a row in 16-byte loads, 8-byte and 4-byte ones, one
# and several passes over the columns; few long buckets, one, as many as rows
# and many more, rows just below and above a team's eight
SHAPES = [(5000, 32, 1024), (5000, 4, 7), (30_000, 64, 100), (30_000, 36, 40_000), (9, 128, 3), (8, 100, 1),
          (70_000, 100, 1), (40_000, 256, 5000), (7, 256, 30), (3000, 260, 900), (20_000, 50, 2500), (2000, 66, 11),
          (1000, 130, 4000), (20_000, 17, 4096), (4097, 33, 33), (3000, 301, 77), (1, 5, 3), (100_000, 8, 20_000)]


@pytest.mark.parametrize("n,d,r", SHAPES)
def test_dense_gather_is_exact(lsk, n, d, r):
    A = integers(n, d, n + d)
    bucket, sign = ocs.countsketch_hash(n, r, 5)
    ref = np.zeros((r, d))
    np.add.at(ref, bucket, A.astype(np.float64) * sign[:, None])
    At = torch.from_numpy(A).cuda()
    for a in (At, torch.cat([At, At[:, :1]], 1)[:, :d], torch.cat([At, At[:, :1], At[:, :1]], 1)[:, :d]):   # strides d .. d + 2
        got = lsk.cs_sketch(a, r, 5).cpu().numpy()
        assert np.array_equal(got.astype(np.float64), ref), (n, d, r, a.stride())


@pytest.mark.parametrize("n,d,r", [(3000, 64, 100), (20_000, 50, 2500), (5000, 256, 9000)])
def test_dense_gather_adds_to_a_sketch(lsk, n, d, r):
    A = integers(n, d, 3)
    At = torch.from_numpy(A).cuda()
    whole = lsk.cs_sketch(At, r, 7).cpu().numpy()
    SA = lsk.sketch_rows(At[:n // 3], r, 0, 7)
    lsk.sketch_rows(At[n // 3:], r, 0, 7, row0=n // 3, out=SA, accumulate=True)
    assert np.array_equal(SA.cpu().numpy(), whole)
