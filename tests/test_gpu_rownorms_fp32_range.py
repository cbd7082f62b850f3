"""FP32 row norms of large dense A: rows outside the range of the tensor-core form
go to the CUDA cores, whatever columns of B their result comes from.  Compared
with the CUDA-core form on the same rows (a call on few rows takes it)."""
import pytest
import torch

pytestmark = pytest.mark.gpu

KINDS = ["general", "odd_zero", "even_zero", "one", "two", "dominant", "dominant_row"]


@pytest.mark.parametrize("kind", KINDS)
def test_rows_outside_the_range(kind):
    import paper_2203_02798_gb300 as lsk
    d, c = 256, {"one": 1, "two": 2}.get(kind, 256)
    n = (1 << 30) // (d * c) + 37          # the smallest that takes the tensor-core form
    g = torch.Generator(device="cuda").manual_seed(7)
    k = torch.arange(n, device="cuda") % 21
    A = torch.randn((n, d), generator=g, device="cuda")
    # one row in 21 each is scaled by 2^0 .. 2^-20 in the first 8,400 rows; the others stand for the typical row
    A[:8400] *= torch.pow(2.0, -k[:8400].float()).view(-1, 1)
    B = torch.randn((d, c), generator=g, device="cuda")
    if kind == "odd_zero":
        B[:, 1::2] = 0.0
    if kind == "even_zero":
        B[:, 0::2] = 0.0
    if kind == "dominant":                 # one column makes the norm, its largest entry meets only zeros
        B[:, 6] *= 1e3
        B[0, 6] = 1e6
        A[:, 0] = 0.0
    if kind == "dominant_row":             # one row of B makes every column but for the (larger) rows with a zero there
        B[0] *= 1e4
        A[:8400] *= torch.pow(4.0, k[:8400].float()).view(-1, 1)
        A[:8400, 0] = 0.0
    x = lsk.rownorms_prod(A, B, prec="fp32")[:8400].double()
    few = lsk.rownorms_prod(A[:2100].contiguous(), B, prec="fp32")
    few = torch.cat([few] + [lsk.rownorms_prod(A[i:i + 2100].contiguous(), B, prec="fp32") for i in (2100, 4200, 6300)]).double()
    want = (A[:8400].double() @ B.double()).square().sum(1)
    rms = lambda v, i: ((v / want - 1.0)[k[:8400] == i]).square().mean().sqrt().item()
    for i in range(21):
        # no more than twice the CUDA-core form's error (a result's rounding, 2^-24, at least)
        assert rms(x, i) <= 2.0 * max(rms(few, i), 2.0 ** -24), (i, rms(x, i), rms(few, i))


def test_zero_and_tiny_rows():
    import paper_2203_02798_gb300 as lsk
    d = c = 256
    n = (1 << 30) // (d * c) + 5
    g = torch.Generator(device="cuda").manual_seed(8)
    A = torch.randn((n, d), generator=g, device="cuda")
    A[::3] = 0.0
    A[1::9] *= 1e-18                       # squares near and below FP32's bottom
    B = torch.randn((d, c), generator=g, device="cuda") / 16.0
    x = lsk.rownorms_prod(A, B, prec="fp32")
    few = torch.cat([lsk.rownorms_prod(A[i:i + 4000].contiguous(), B, prec="fp32") for i in range(0, n, 4000)])
    assert torch.equal(x[::3], torch.zeros_like(x[::3]))
    assert torch.allclose(x, few, rtol=2e-6, atol=0.0)



@pytest.mark.parametrize("n,d", [(70_000, 128), (262_144, 64), (20_000, 256), (33_000, 200)])
def test_error_of_inverse_factors(n, d):
    """x = ||A_i R^-1||^2 with A's own R, as the leverage scores form them: no
    further off than on the CUDA cores (3% for the spread of the mean over n rows)."""
    import paper_2203_02798_gb300 as lsk
    g = torch.Generator(device="cuda").manual_seed(10)
    A = torch.randn((n, d), generator=g, device="cuda")
    R = torch.linalg.qr(A.double(), mode="r")[1]
    B = torch.linalg.solve_triangular(R, torch.eye(d, dtype=torch.float64, device="cuda"), upper=True).float().contiguous()
    step = (1 << 30) // (d * d) - 1        # rows of a call that takes the CUDA cores
    x = lsk.rownorms_prod(A, B, upper_triangular=True, prec="fp32").double()
    few = torch.cat([lsk.rownorms_prod(A[i:i + step].contiguous(), B, upper_triangular=True, prec="fp32")
                     for i in range(0, n, step)]).double()
    want = (A.double() @ B.double()).square().sum(1)
    rms = lambda v: (v / want - 1.0).square().mean().sqrt().item()
    assert rms(x) <= 1.03 * rms(few)


def stage_times(lsk, A, B):
    """x, and the time of the tensor-core pass and of the CUDA-core pass behind it (ms)."""
    lsk.rownorms_prod(A, B, prec="fp32")
    ctx = lsk.context()
    ctx.profile_reset()
    ctx.profile(True)
    x = lsk.rownorms_prod(A, B, prec="fp32")
    ctx.sync()
    times = ctx.profile_totals()
    ctx.profile(False)
    return x, times["rownorm_dense_tc3"][1], times["rownorm_dense_simt"][1]


@pytest.mark.parametrize("c", [96, 256])
@pytest.mark.parametrize("kind", ["zero_column", "rare_column", "first_columns_zero", "mostly_small_rows", "mostly_zero_rows"])
def test_work_shared_by_the_sample(kind, c):
    """Columns that the sampled rows do not show leave the rows on the tensor
    cores; where most rows are outside the range, the CUDA cores do all of them
    and the tensor-core pass ends at once."""
    import paper_2203_02798_gb300 as lsk
    n, d = 300_000, 96
    g = torch.Generator(device="cuda").manual_seed(9)
    A = torch.randn((n, d), generator=g, device="cuda") * torch.logspace(-2, 2, d, device="cuda")
    B = torch.randn((d, c), generator=g, device="cuda")
    if kind == "zero_column":
        A[:, 50] = 0.0
    if kind == "rare_column":
        A[:, 3] = 0.0
        A[1234::100_000, 3] = 1.0
    if kind == "first_columns_zero":
        A[:, :40] = 0.0
    if kind == "mostly_small_rows":
        A[torch.arange(n, device="cuda") % 8 != 3] *= 1e-5
    if kind == "mostly_zero_rows":
        A[torch.arange(n, device="cuda") % 8 != 3] = 0.0
    x, tc, simt = stage_times(lsk, A, B)
    want = (A.double() @ B.double()).square().sum(1)
    bound = (2 * (d + 2) + c + 4) * 2.0 ** -24 * ((A.double().abs() @ B.double().abs()).square().sum(1))
    assert torch.all((x.double() - want).abs() <= bound)
    assert (tc < 0.3 * simt) if kind == "mostly_small_rows" else (simt < tc)


@pytest.mark.parametrize("beta", [0.0, 0.5])
@pytest.mark.parametrize("listed", [1, 5, 156, 158, 627, 629, 1500])
def test_few_listed_rows(listed, beta):
    """The CUDA cores' forms for few listed rows (up to four a block of the 157
    tiles here) and for more: the rows that a call on them alone gives."""
    import paper_2203_02798_gb300 as lsk
    n, d = 20_001, 256
    g = torch.Generator(device="cuda").manual_seed(11)
    A = torch.randn((n, d), generator=g, device="cuda")
    at = torch.arange(listed, device="cuda") * (n // listed)
    A[at] *= 2.0 ** -14
    B = torch.triu(torch.randn((d, d), generator=g, device="cuda"))
    x0 = torch.rand(n, generator=g, device="cuda")
    x = lsk.rownorms_prod(A, B, alpha=2.0, beta=beta, x=x0.clone(), upper_triangular=True, prec="fp32").double()
    want = 2.0 * (A.double() @ B.double()).square().sum(1) + beta * x0.double()
    size = 2.0 * (A.double().abs() @ B.double().abs()).square().sum(1) + beta * x0.double()
    assert torch.all((x - want).abs() <= 2 * (d + 4) * 2.0 ** -24 * size)


def test_few_listed_rows_cost_little():
    import paper_2203_02798_gb300 as lsk
    n, d = 33_000, 256
    A = torch.randn((n, d), generator=torch.Generator(device="cuda").manual_seed(12), device="cuda")
    A[::10_000] *= 2.0 ** -14
    x, tc, simt = stage_times(lsk, A, torch.eye(d, device="cuda"))
    assert simt < 0.5 * tc
