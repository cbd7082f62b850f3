"""CountSketch of CSR A: the error of its sums against 64 bits, by the number of
nonzeros that meet in an entry."""
import numpy as np
import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r", [1024, 4096, 20_000])
@pytest.mark.parametrize("per_entry", [0.4, 2.0, 6.0, 14.0])
def test_error_of_sums(r, per_entry):
    """A chain of k additions of terms of random sign grows as a random walk and is
    off by 2^-24 x 0.3 sqrt(k) of its size (a rounding 0.29 ulp, an ulp 0.72 x 2^-23 in
    the mean); with k Poisson of mean c, weighted by size, 0.3 sqrt(c + 2).  A bucket
    of few may be split in P parts, whose sums are then added up.  The better of the
    two, with a tenth for the estimate."""
    import paper_2203_02798_gb300 as lsk
    n, d = 200_000, 64
    P = 1
    while P < 32 and r * P < 16384 and n >= r * P * 8:
        P *= 2
    V, J, I = workloads.csr_bernoulli(n, d, per_entry * r / n, seed=r)
    SA = lsk.cs_sketch(lsk.csr_from_numpy(V, J, I, d), r, 17).cpu().numpy().astype(np.float64)
    h, s = lsk.debug_hash(n, r, 17)
    rows = np.repeat(np.arange(n), np.diff(I))
    at = h.cpu().numpy()[rows].astype(np.int64) * d + J
    want = np.bincount(at, weights=V.astype(np.float64) * s.cpu().numpy()[rows], minlength=r * d).reshape(r, d)
    k = min(per_entry + 2, per_entry / P + 2 + P + 2)
    assert np.linalg.norm(SA - want) <= 2.0 ** -24 * 0.33 * k ** 0.5 * np.linalg.norm(want)


@pytest.mark.parametrize("n,d,r,nz", [(70_000, 64, 4096, 20), (9000, 17, 1000, 9), (200_000, 100, 10_000, 30),
                                      (140_000, 256, 16_383, 40), (200_000, 100, 10_000, 3)])
def test_copies_are_exact_on_whole_numbers(n, d, r, nz):
    """Sums of small whole numbers, exact in any order, in the callers of the form
    with two and four copies: alone, and added to a sketch."""
    import paper_2203_02798_gb300 as lsk
    rng = np.random.default_rng(n)
    I = np.arange(n + 1, dtype=np.int64) * nz
    J = rng.integers(0, d, size=n * nz).astype(np.int32)
    V = rng.integers(-4, 5, size=n * nz).astype(np.float32)
    A = lsk.csr_from_numpy(V, J, I, d)
    h, s = lsk.debug_hash(n, r, 5)
    rows = np.repeat(np.arange(n), nz)
    at = h.cpu().numpy()[rows].astype(np.int64) * d + J
    want = np.bincount(at, weights=V.astype(np.float64) * s.cpu().numpy()[rows], minlength=r * d).reshape(r, d)
    for _ in range(2):
        assert np.array_equal(lsk.cs_sketch(A, r, 5).cpu().numpy(), want)
    out = torch.ones((r, d), dtype=torch.float32, device="cuda")
    lsk.sketch_rows(A, r, 0, 5, "fp32", 0, out=out, accumulate=True)
    lsk.context().sync()
    assert np.array_equal(out.cpu().numpy(), want + 1.0)
