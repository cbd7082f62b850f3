"""FP32 Gram matrix on the tensor cores: the units of its split come from a sample
of the rows, from which no pattern of rows hides."""
import pytest
import torch

pytestmark = pytest.mark.gpu
U24 = 2.0 ** -24


def exact(A):
    C = torch.zeros((A.shape[1],) * 2, dtype=torch.float64, device="cuda")
    for i in range(0, A.shape[0], 1 << 18):
        b = A[i:i + (1 << 18)].double()
        C += b.T @ b
    return C


@pytest.mark.parametrize("n,d", [(250_003, 64), (1_000_000, 200)])
@pytest.mark.parametrize("period,at", [(8, 5), (8, 2), (32, 13), (128, 77)])
def test_periodic_columns(n, d, period, at):
    """Every third column is nonzero in one row of a period only: within 4 x 2^-24 of
    sqrt(C_aa C_bb), as for any A."""
    import paper_2203_02798_gb300 as lsk
    A = torch.randn((n, d), generator=torch.Generator(device="cuda").manual_seed(6), device="cuda")
    A[:, ::3] *= (torch.arange(n, device="cuda") % period == at).float().view(-1, 1)
    C = exact(A)
    s = C.diagonal().sqrt()
    assert torch.all((lsk.gram(A, prec="fp32").double() - C).abs() <= 4 * U24 * torch.outer(s, s))


@pytest.mark.parametrize("first,rest", [(0.0, 1.0), (1e-3, 1.0), (1.0, 1e-3), (1e3, 0.0)])
def test_columns_that_change(first, rest):
    """Columns that are zero, small or large in the first rows of a CTA, then not."""
    import paper_2203_02798_gb300 as lsk
    n, d = 600_000, 96
    A = torch.randn((n, d), generator=torch.Generator(device="cuda").manual_seed(7), device="cuda")
    A[:, ::2] *= torch.where(torch.arange(n, device="cuda") % 3000 < 700, first, rest).float().view(-1, 1)
    C = exact(A)
    s = C.diagonal().sqrt()
    assert torch.all((lsk.gram(A, prec="fp32").double() - C).abs() <= 4 * U24 * torch.outer(s, s))
