"""FP32 Gram matrix of very tall A (lsk_gram_prec FP32 on the tensor cores): the
error does not grow with the number of rows."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,d", [(16_000_003, 64), (5_000_000, 200), (4_000_000, 256)])
def test_error_of_many_rows(n, d):
    """Storing C in FP32 has an error of its own (about 1.8e-8 in the norm); the
    sums before it are 24 additions long at most, each rounded to 2^-24 (0.29 of
    2^-23 in the mean), and averaged over the CTAs' partials, some 300 or more:
    6e-9, which adds in the square."""
    import paper_2203_02798_gb300 as lsk
    A = torch.randn((n, d), generator=torch.Generator(device="cuda").manual_seed(5), device="cuda")
    A.mul_(0.01).add_(1.0)
    C = torch.zeros((d, d), dtype=torch.float64, device="cuda")
    for i in range(0, n, 1 << 18):
        b = A[i:i + (1 << 18)].double()
        C += b.T @ b
    got = lsk.gram(A, prec="fp32").double()
    size = torch.linalg.norm(C)
    stored = (torch.linalg.norm(C.float().double() - C) / size).item()
    assert (torch.linalg.norm(got - C) / size).item() <= (stored ** 2 + 6e-9 ** 2) ** 0.5
