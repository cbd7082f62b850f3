"""Row norms of dense A on the CUDA cores: calls that follow one another directly
take no longer than calls with another kernel between them, which lets none of the
next in early."""
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


@pytest.mark.parametrize("n,d,c", [(10_000, 400, 64), (30_000, 600, 64), (50_000, 400, 64), (50_000, 400, 128)])
def test_a_call_does_not_hinder_the_one_before(n, d, c):
    import paper_2203_02798_gb300 as lsk
    g = torch.Generator(device="cuda").manual_seed(1)
    A = torch.randn((n, d), generator=g, device="cuda")
    B = torch.randn((d, c), generator=g, device="cuda")
    z = torch.zeros(16, device="cuda")

    def apart():
        z.add_(1)
        lsk.rownorms_prod(A, B)

    assert _ms(lambda: lsk.rownorms_prod(A, B), 20) <= 1.1 * _ms(apart, 20)
