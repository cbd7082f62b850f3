"""Row norms of CSR A: the time follows the nonzeros where rows are few and dense,
and the norms are FP32's for any number of rows a warp."""
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
    B = torch.randn((100, 100), generator=torch.Generator(device="cuda").manual_seed(2), device="cuda")
    few, more = _csr(3_000, 100, 23)[0], _csr(100_000, 100, 23)[0]
    assert _ms(lambda: lsk.rownorms_prod(few, B)) <= 0.5 * _ms(lambda: lsk.rownorms_prod(more, B))


# 32, 16, 8 and 4 rows a warp; short last groups
@pytest.mark.parametrize("n,d,per", [(1, 64, 40), (5, 40, 33), (127, 64, 4), (3_001, 100, 5), (3_001, 100, 9),
                                     (4_999, 100, 23), (200_003, 32, 4)])
def test_against_fp64(n, d, per):
    import paper_2203_02798_gb300 as lsk
    A, V, J = _csr(n, d, per)
    B = torch.randn((d, d), generator=torch.Generator(device="cuda").manual_seed(2), device="cuda")
    M = B.double() @ B.double().T
    V, J = V.double().view(n, per), J.long().view(n, per)
    want = torch.zeros(n, dtype=torch.float64, device="cuda")
    mags = torch.zeros_like(want)
    Mags = B.double().abs() @ B.double().abs().T
    for p in range(per):
        for t in range(per):
            want += V[:, p] * V[:, t] * M[J[:, p], J[:, t]]
            mags += (V[:, p] * V[:, t]).abs() * Mags[J[:, p], J[:, t]]
    # d additions in an entry of M, per in an entry's sum, per in the row's, one rounding each, and the products'
    bound = (d + 2 * per + 4) * 2.0**-24 * mags
    assert ((lsk.rownorms_prod(A, B).double() - want).abs() <= bound + 1e-30).all()
