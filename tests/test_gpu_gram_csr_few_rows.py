"""A^T A of CSR A with few but dense rows: the time follows the nonzeros, and the
result is FP32's, when several warps share a group of rows."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _ms(run, reps=10):
    for _ in range(4):
        run()
    best = float("inf")
    for _ in range(7):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        for _ in range(reps):
            run()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) / reps)
    return best


def _csr(n, d, per):
    import paper_2203_02798_gb300 as lsk
    g = torch.Generator(device="cuda").manual_seed(1)
    I = per * torch.arange(n + 1, dtype=torch.int64, device="cuda")
    J = torch.randint(0, d, (n * per,), generator=g, device="cuda", dtype=torch.int32)
    V = torch.randn(n * per, generator=g, device="cuda")
    return lsk.CSR(V, J, I, n, d), V, J


def test_time_follows_the_nonzeros():
    import paper_2203_02798_gb300 as lsk
    few, more = _csr(10_000, 256, 50)[0], _csr(50_000, 256, 50)[0]
    assert _ms(lambda: lsk.gram(few)) <= 0.6 * _ms(lambda: lsk.gram(more))


# 1, 2, 4, ... warps a group of 32 rows; rows of one group and none; a short last group
@pytest.mark.parametrize("n,d,per", [(1, 256, 50), (31, 300, 40), (33, 256, 200), (3_001, 230, 20), (10_000, 256, 50),
                                     (10_000, 400, 3), (40_001, 250, 12), (200_000, 256, 13)])
def test_against_fp64(n, d, per):
    import paper_2203_02798_gb300 as lsk
    A, V, J = _csr(n, d, per)
    D = torch.zeros((n, d), dtype=torch.float64, device="cuda")
    rows = torch.arange(n, device="cuda").repeat_interleave(per)
    D.index_put_((rows, J.long()), V.double(), accumulate=True)   # a column twice in a row adds up
    want = D.T @ D
    mags = torch.zeros_like(D)
    mags.index_put_((rows, J.long()), V.double().abs(), accumulate=True)
    # an entry is a sum of up to about 10,000 products in FP32, whose roundings walk at
    # random: 64 times a rounding of the sum of the magnitudes, chains of no more than 100
    # on their way through blocks, copies and the sum of the copies
    bound = 64 * 2.0**-24 * (mags.T @ mags)
    assert ((lsk.gram(A).double() - want).abs() <= bound + 1e-30).all()
