"""Row norms of CSR A on the GPU alone (replayed, so that no launch is waited for):
a lane a row and a lane a nonzero, each where it is the faster."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _replay_ms(n, d, per, calls=20):
    import paper_2203_02798_gb300 as lsk
    g = torch.Generator(device="cuda").manual_seed(1)
    I = per * torch.arange(n + 1, dtype=torch.int64, device="cuda")
    nnz = n * per
    J = torch.randint(0, d, (nnz,), generator=g, device="cuda", dtype=torch.int32)
    A = lsk.CSR(torch.randn(nnz, generator=g, device="cuda"), J, I, n, d)
    B = torch.randn((d, 16), generator=g, device="cuda")
    for _ in range(3):
        lsk.rownorms_prod(A, B)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for _ in range(calls):
            lsk.rownorms_prod(A, B)
    best = float("inf")
    for _ in range(9):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        graph.replay()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) / calls)
    return best


def test_few_columns_keep_a_lane_a_row():
    # five nonzeros a row: one read of M's 9 columns a pair against finding the entries
    assert _replay_ms(200_000, 9, 5) <= 0.7 * _replay_ms(200_000, 64, 5)
