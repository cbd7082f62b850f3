"""Row norms of CSR A on the GPU alone (replayed, so that no launch is waited for):
short rows of mixed lengths."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _replay_ms(n, d, per, calls=20):
    import paper_2203_02798_gb300 as lsk
    g = torch.Generator(device="cuda").manual_seed(1)
    lengths = torch.poisson(torch.full((n,), per, device="cuda"), generator=g).long()
    I = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    I[1:] = torch.cumsum(lengths, 0)
    nnz = int(I[-1])
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


def test_time_beside_denser_rows():
    # three nonzeros a row in the mean, a lane a row; 5.5, a lane a nonzero
    assert _replay_ms(53_322, 256, 3.0) <= 1.2 * _replay_ms(53_322, 256, 5.5)
